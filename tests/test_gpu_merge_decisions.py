"""The merge's choice of a target, token by token (read from the call's workspace), on inputs whose answer is known
by construction: sums that need all of the lanes' fp64 addition, several targets that the tensor core's product
cannot tell apart, products that its accumulation drops, tokens so small that their norm underflows, copies of
targets; and the accumulation error that the screening's bound rests on."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def assigned(riftlib, cuda, X, m, N=1):
    """The target index (0 .. m - 1) of every unselected token of one tile X [n_v, d] whose token 0 is selected, with m
    targets: tokens 1, 1 + R // m, ...  A target's own entry is left as it was (-1).  The tile is the last of N."""
    n_v, d = X.shape
    i32 = dict(dtype=torch.int32, device=cuda)
    sel = torch.zeros(n_v, **i32)
    ctx = torch.zeros(m, d, dtype=torch.bfloat16, device=cuda)
    ctx_target = torch.zeros(m, **i32)
    need = riftlib.merge_workspace_bytes(N, n_v)
    ws = torch.full((need,), 255, dtype=torch.uint8, device=cuda)
    xdt = riftlib.RIFT_BF16 if X.dtype == torch.bfloat16 else riftlib.RIFT_F32
    tiles = torch.zeros(N, n_v, d, dtype=X.dtype, device=cuda)
    tiles[N - 1] = X.to(cuda)
    sel_off, kept = torch.ones(N + 1, **i32), torch.full((N,), N - 1, **i32)
    sel_off[0] = 0
    ctx_off = torch.zeros(N + 1, **i32)
    riftlib.merge_contextual(tiles, xdt, N, n_v, d, kept, torch.ones(1, **i32), torch.full((N,), 1 + m, **i32), sel, sel_off,
                             ctx, m, ctx_off, ctx_target, ws, need)
    riftlib.sync_status()
    R = n_v - 1
    step = R // m
    assert ctx_target.cpu().tolist() == [1 + q * step for q in range(m)]
    off = (N * n_v * 4 + 255) // 256 * 256  # the unselected tokens' list, then the assignment
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


def one_hot(d, **at):
    """A row of zeros but for c<column>=value."""
    v = torch.zeros(d)
    for k, e in at.items():
        v[int(k[1:])] = e
    return v


# targets that differ from 1 by a product of 2^-26 or less with their token, which an accumulation with 1 drops: the
# screening sees them as equal.  Up to 7: the candidates are listed; more, or more than 2 beyond the 80 targets of
# one block: all targets are looked at; d above and off a warp's 256-column steps.  fp32 tokens, whose sums drop the
# products too: a third near target has all looked at
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32], ids=["bf16", "f32"])
@pytest.mark.parametrize("near,m", [(2, 2), (3, 6), (4, 6), (7, 9), (8, 9), (7, 80), (80, 80), (2, 81), (3, 81), (100, 100)])
@pytest.mark.parametrize("d", [320, 4096])
def test_best_of_several_near_targets(near, m, d, dtype, cuda, riftlib):
    targets = [one_hot(d, c0=1.0, **{f"c{2 + q}": 2.0 ** -14}) if q < near else one_hot(d, **{f"c{2 + q}": 1.0})
               for q in range(m)]
    wins = sorted({0, 1, near // 2, near - 1})
    tokens = []
    for w in wins:  # 2^-13 against 2^-14 at the winner's own column: products 2^-27 and 2^-28
        x = one_hot(d, c0=1.0)
        for q in range(near):
            x[2 + q] = 2.0 ** -13 if q == w else 2.0 ** -14
        tokens.append(x)
    tokens.append(one_hot(d, c0=1.0))  # an exact tie: the lowest
    X, at = tile(d, targets, tokens, dtype)
    got = assigned(riftlib, cuda, X, m)
    assert [got[a] for a in at] == wins + [0]


# products of 1.98 x 2^-26 in every other column, all dropped next to 1, against one of a kept size that is worth a
# little less than their sum: the product ranks the targets the wrong way round by about as much as it can
@pytest.mark.parametrize("scale", [0, -40, -100], ids=["one", "small", "tiny"])  # 2^-200: the squares underflow
@pytest.mark.parametrize("d", [64, 512, 4096, 8192])
def test_dropped_products_do_not_decide(d, scale, cuda, riftlib):
    s = 1.40625  # s^2 = 1.9775, 8 bits
    many = list(range(2, d, 2))
    a, b = torch.zeros(d), torch.zeros(d)
    a[0] = b[0] = 1.0
    a[many] = s * 2.0 ** -13
    b[[k - 1 for k in many]] = s * 2.0 ** -13  # the same norm
    x = torch.zeros(d)
    x[0] = 1.0
    x[many] = s * 2.0 ** -13
    total = len(many) * s * s * 2.0 ** -26
    x[1] = (0.95 * total / b[1]).to(torch.bfloat16)
    exact = [float(x.double() @ t.double()) for t in (b, a)]
    assert exact[1] > exact[0] > 1 and float(x[1] * b[1]) > 2.0 ** -25
    X, at = tile(d, [b, a], [x * 2.0 ** scale, x * 2.0 ** scale], torch.bfloat16)
    got = assigned(riftlib, cuda, X, 2)
    assert [got[k] for k in at] == [1, 1]


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32], ids=["bf16", "f32"])
def test_blank_tokens_and_copies_of_targets(dtype, cuda, riftlib):
    """Blank rows (all alike, or zero) make many targets copies of one: a blank token goes to the first of them, a zero
    one to the first target."""
    d, m = 256, 9
    g = torch.Generator()
    g.manual_seed(3)
    blank, zero = torch.randn(d, generator=g), torch.zeros(d)
    other = [torch.randn(d, generator=g) for _ in range(4)]
    targets = [other[0], blank, blank, zero, other[1], blank, other[2], zero, blank]
    tokens = [blank, zero, other[1], -blank, blank, zero, other[2], blank + 0, other[0]]
    X, at = tile(d, targets, tokens, dtype)
    x64, t64 = X.double(), torch.stack(targets).to(dtype).double()
    nrm = t64.norm(dim=1, keepdim=True)
    unit = torch.where(nrm > 0, t64 / nrm.clamp_min(1e-300), t64)
    want = [int((unit @ x64[1 + a]).argmax()) for a in at]
    want = [1 if w in (1, 2, 5, 8) else w for w in want]  # equal rows tie in exact arithmetic: the lower
    assert want[0] == 1 and want[1] == 0 and want[2] == 4
    got = assigned(riftlib, cuda, X, m)
    assert [got[a] for a in at] == want


def test_fp32_assignment_does_not_depend_on_the_tile_count(cuda, riftlib):
    """fp32 tokens: the forms for few and for many tiles (204 tiles of 9 token blocks) choose alike, tokens between
    many near-duplicate targets among them."""
    n_v, d, m = 576, 320, 37
    g = torch.Generator()
    g.manual_seed(5)
    X = torch.randn(n_v, d, generator=g)
    X[1::3] = X[1] + 1e-3 * torch.randn(len(X[1::3]), d, generator=g)  # all targets among them
    few, many = (assigned(riftlib, cuda, X, m, N) for N in (1, 204))
    assert few == many
    x = X.double()
    step = (n_v - 1) // m
    unit = x[1:1 + m * step:step] / x[1:1 + m * step:step].norm(dim=1, keepdim=True)
    want = (x[1:] @ unit.T).argmax(dim=1).tolist()
    for a in range(n_v - 1):
        if a % step or a // step >= m:
            assert few[a] == want[a], a


@pytest.mark.parametrize("K", [64, 256, 4096])
@pytest.mark.parametrize("sign", [1, -1])
def test_accumulation_error_per_update(K, sign, cuda, riftlib):
    """What the screening's bound takes for granted, on the same accumulators through rift_linear's fp32 epilogue: an
    update of 16 products and the accumulator loses less than 2^-25 of the largest addend an addend, and 2^-23 of the
    result.  Addends next to a 1: every power of two from 2^-18 to 2^-30, times 1 and times 1.98."""
    M, N = 64, 64
    A, W = torch.zeros(M, K), torch.zeros(N, K)
    A[:, 0] = W[:, 0] = 1.0
    for r in range(26):
        e, f = 18 + r // 2, 1.40625 if r % 2 else 1.0
        A[r, 1:] = f * 2.0 ** -(e // 2)
    W[:32, 1:] = sign * 2.0 ** -9
    W[32:, 1:] = sign * 1.40625 * 2.0 ** -9
    A, W = A.to(torch.float16), W.to(torch.float16)
    R = torch.zeros(M, N, device=cuda)
    riftlib.linear(A.to(cuda), W.to(cuda), M, N, K, riftlib.RIFT_EPI_RESID_F32, R)
    riftlib.sync_status()
    exact = A.double() @ W.double().T
    largest = (A.double().norm(dim=1)[:, None] * W.double().norm(dim=1)[None])
    # K / 16 updates of 16 addends; K may be split and its parts added in fp32 (8 of them at most)
    bound = (K / 16 * (16 * 2.0 ** -25 + 2.0 ** -23) + 8 * 2.0 ** -24) * largest
    assert bool(((R.cpu().double() - exact).abs() <= bound).all())
