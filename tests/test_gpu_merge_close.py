"""The merge's choice between close targets (bf16 tokens): the tensor-core screening decides alone only
where its best target is clear of the others by more than its error bound, everything else is
decided by float-float sums.  Tiles of near-duplicate tokens (cosine gaps from 1e-2 down to 1e-8) and
exact duplicates (ties to the lower target), one, few and more than 128 targets per slot: every token's
assignment, as the call leaves it in its workspace, against the oracle's groups, and the groups' means."""
import pytest
import torch

from oracle import rift_oracle as O
from synth import rng

pytestmark = pytest.mark.gpu


def _tile(n_v, d, protos, step_bits, seed):
    """Token k = prototype k mod protos with a few elements moved by 2^-step_bits of their value;
    every fifth token is the prototype itself."""
    p = rng.normal_f32(seed, rng.stream_id("close-proto"), protos * d).view(protos, d)
    z = rng.normal_f32(seed, rng.stream_id("close-noise"), n_v * d).view(n_v, d)
    x = p[torch.arange(n_v) % protos].clone()
    moved = z.abs() > 1.5
    moved[::5] = False
    x = torch.where(moved, x * (1 + torch.sign(z) * 2.0 ** -step_bits), x)
    return x.to(torch.bfloat16)


@pytest.mark.parametrize("n_v,d,m,protos,bits", [(576, 512, 45, 20, 3), (576, 512, 45, 20, 6), (600, 256, 150, 40, 5),
                                                 (130, 4096, 20, 9, 7), (72, 64, 1, 3, 4), (576, 8192, 30, 500, 2)])
def test_close_targets(n_v, d, m, protos, bits, cuda, riftlib):
    X = torch.stack([_tile(n_v, d, protos, bits, s) for s in (1, 2)])
    dom = [[k for k in range(n_v) if (3 * k + t) % 7 == 0] for t in range(2)]  # the selected tokens
    ref = [O.merge_contextual(X[t], dom[t], m) for t in range(2)]
    for t, (targets, groups, _) in enumerate(ref):  # the decisions are unique at the rescoring's accuracy
        xt = X[t][targets].double()
        xt = xt / xt.norm(dim=1, keepdim=True)
        for j, gr in enumerate(groups):
            sims = xt @ X[t][gr].double().T / X[t][gr].double().norm(dim=1)
            same = (xt == xt[j]).all(dim=1)
            gap = (sims[j] - torch.where(same[:, None], -2.0, sims).max(dim=0).values)[1:]
            assert len(gap) == 0 or float(gap.min()) > 1e-10
    i32 = dict(dtype=torch.int32, device=cuda)
    off = [0, len(dom[0]), len(dom[0]) + len(dom[1])]
    sel = torch.zeros(2 * n_v, **i32)
    sel[:off[2]] = torch.tensor(dom[0] + dom[1], **i32)
    ctx = torch.zeros(2 * m, d, dtype=torch.bfloat16, device=cuda)
    ctx_off, ctx_target = torch.zeros(3, **i32), torch.zeros(2 * m, **i32)
    need = riftlib.merge_workspace_bytes(2, n_v)
    ws = torch.empty(need, dtype=torch.uint8, device=cuda)
    riftlib.merge_contextual(X.to(cuda), riftlib.RIFT_BF16, 2, n_v, d, torch.tensor([0, 1], **i32),
                             torch.tensor([2], **i32), torch.tensor([len(dom[0]) + m, len(dom[1]) + m], **i32), sel,
                             torch.tensor(off, **i32), ctx, 2 * m, ctx_off, ctx_target, ws, need)
    riftlib.sync_status()
    assert ctx_off.cpu().tolist() == [0, m, 2 * m]
    off = (2 * n_v * 4 + 255) // 256 * 256  # the unselected tokens' lists, then the assignments
    assign = ws[off:off + 2 * n_v * 4].view(torch.int32).view(2, n_v).cpu()
    for t, (targets, groups, mean) in enumerate(ref):
        rest = [k for k in range(n_v) if k not in set(dom[t])]
        want = {k: q for q, gr in enumerate(groups) for k in gr[1:]}
        assert len(want) == len(rest) - m
        wrong = [(k, int(assign[t, a]), want[k]) for a, k in enumerate(rest) if k in want and int(assign[t, a]) != want[k]]
        assert not wrong, (t, len(wrong), wrong[:5])
        assert ctx_target[t * m:(t + 1) * m].cpu().tolist() == targets
        got = ctx[t * m:(t + 1) * m].cpu().double()
        assert bool(((got - mean).abs() <= mean.abs().clamp_min(1e-30) * 2.0 ** -7).all()), t
