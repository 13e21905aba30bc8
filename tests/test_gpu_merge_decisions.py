"""The merge's choice of a target, token by token (read from the call's workspace), on inputs whose answer is known
by construction: sums that need all of the lanes' fp64 addition."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def assigned(riftlib, cuda, X, m):
    """The target index (0 .. m - 1) of every unselected token of one tile X [n_v, d] whose token 0 is selected, with m
    targets: tokens 1, 1 + R // m, ...  A target's own entry is left as it was (-1)."""
    n_v, d = X.shape
    i32 = dict(dtype=torch.int32, device=cuda)
    sel = torch.zeros(n_v, **i32)
    ctx = torch.zeros(m, d, dtype=torch.bfloat16, device=cuda)
    ctx_off, ctx_target = torch.zeros(2, **i32), torch.zeros(m, **i32)
    need = riftlib.merge_workspace_bytes(1, n_v)
    ws = torch.full((need,), 255, dtype=torch.uint8, device=cuda)
    xdt = riftlib.RIFT_BF16 if X.dtype == torch.bfloat16 else riftlib.RIFT_F32
    riftlib.merge_contextual(X[None].contiguous().to(cuda), xdt, 1, n_v, d, torch.zeros(1, **i32), torch.ones(1, **i32),
                             torch.tensor([1 + m], **i32), sel, torch.tensor([0, 1], **i32), ctx, m, ctx_off, ctx_target,
                             ws, need)
    riftlib.sync_status()
    R = n_v - 1
    step = R // m
    assert ctx_target.cpu().tolist() == [1 + q * step for q in range(m)]
    off = (n_v * 4 + 255) // 256 * 256  # the unselected tokens' list, then the assignment
    return ws[off:off + 4 * R].view(torch.int32).cpu().tolist()


def tile(d, targets, tokens, dtype):
    """Selected token, then each target followed by its share of the tokens (step - 1 of them, padded with copies of the
    last); returns the tile and the positions of the tokens among the unselected."""
    m = len(targets)
    step = -(-len(tokens) // m) + 1
    rows, at, k = [torch.ones(d)], [], 0
    for t in targets:
        rows.append(t)
        for _ in range(step - 1):
            if k < len(tokens):
                at.append(len(rows) - 1)
            rows.append(tokens[min(k, len(tokens) - 1)])
            k += 1
    return torch.stack(rows).to(dtype), at


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32], ids=["bf16", "f32"])
@pytest.mark.parametrize("d", [512, 4096])
def test_lane_sums_keep_fp64(d, dtype, cuda, riftlib):
    """x.t1 = 1 + 2^-24 + 2^-50 against x.t0 = 1 + 2^-24, the terms in different lanes and the norms equal: the sum of
    the lanes' pairs needs 51 bits.  The mirrored token is an exact tie and goes to the lower target."""
    def vec(**at):
        v = torch.zeros(d)
        for k, e in at.items():
            v[int(k[1:])] = 2.0 ** e
        return v
    # 8 elements per lane: columns 0, 8, 16, 24 belong to lanes 0, 1, 2, 3
    t0 = vec(c0=0, c8=-12, c24=-25)
    t1 = vec(c0=0, c8=-12, c16=-25)
    x = vec(c0=0, c8=-12, c16=-25)
    tie = vec(c0=0, c8=-12, c32=-25)
    y = vec(c0=0, c8=-12, c24=-25)
    X, at = tile(d, [t0, t1], [x, tie, y, x], dtype)
    got = assigned(riftlib, cuda, X, 2)
    assert [got[a] for a in at] == [1, 0, 0, 1]
