"""The selection in one launch (up to 512 tiles) at the edges of its range and of a thread's tiles, and the
two launches above it, against the oracle on shared fp32 inputs: integers and normalised scores exactly."""
import numpy as np
import pytest
import torch

from oracle import rift_oracle as O
from synth import rng
from synth import workloads as W

pytestmark = pytest.mark.gpu

POLICY = W.Policy(0.3, (1, 8, 16, 64), (0.9, 0.9, 0.9, 0.9), (0.2, 0.5, 0.7, 0.9), (0.1, 0.2, 0.4, 1.0), 0.2)


@pytest.mark.parametrize("ext_p", [False, True], ids=["own", "ext_p"])
@pytest.mark.parametrize("N,n_v", [(1, 64), (4, 65), (5, 576), (256, 64), (257, 100), (511, 65), (512, 64), (513, 64), (1023, 64), (1024, 70), (1025, 64)])
def test_selection_matches_the_oracle(N, n_v, ext_p, cuda, riftlib):
    r = rng.normal_f32(8, rng.stream_id("select-one", N), N * n_v).view(N, n_v)
    r = torch.floor(r * 16) / 16  # ties
    s = rng.normal_f32(8, rng.stream_id("select-one-s", N), N)
    p = rng.uniform_f32(8, 99, N) if ext_p else None
    dev = dict(dtype=torch.int32, device=cuda)
    u = torch.empty(N, device=cuda)
    kept, n_kept, bud = torch.empty(N, **dev), torch.empty(1, **dev), torch.empty(N, **dev)
    sel, off = torch.full((N * n_v,), -1, **dev), torch.empty(N + 1, **dev)
    riftlib.select_budgeted_tokens(r.to(cuda), s.to(cuda), N, n_v, p.to(cuda) if ext_p else None,
                                   riftlib.make_policy(POLICY), u, kept, n_kept, bud, sel, off, None, 0)
    riftlib.sync_status()
    r32, s32 = r.numpy().astype(np.float32), s.numpy().astype(np.float32)
    ou = O.minmax_normalize(s32)
    ok = O.retained(ou, POLICY.tau)
    ob = [O.budget(float(np.float32(p[i]) if ext_p else ou[i]), POLICY) for i in ok]
    assert np.array_equal(u.cpu().numpy().view(np.uint32), ou.view(np.uint32))
    n = int(n_kept.item())
    assert kept[:n].cpu().tolist() == ok and bud[:n].cpu().tolist() == ob
    o = off.cpu().tolist()
    assert o[:n + 1] == [0] + list(np.cumsum(ob)) and all(v == sum(ob) for v in o[n:])
    g = sel.cpu().tolist()
    for j, i in enumerate(ok):
        assert g[o[j]:o[j + 1]] == O.top_b(r32[i], ob[j])


@pytest.mark.parametrize("N,n_v,C", [(512, 1024, 1024), (512, 576, 72), (1024, 1024, 1024), (1024, 576, 72), (1023, 1024, 1024), (256, 64, 64)])
def test_every_tile_kept(N, n_v, C, cuda, riftlib):
    """Equal scores keep every tile (u = 1): the largest tile count the scan over kept tiles and their
    tokens has to hold, at the largest token count and at a smaller one."""
    pol = W.Policy(1.0, (C,), (0.9,), (0.2,), (0.1,), 0.2)
    r = (torch.arange(N * n_v) * 7919 % 1009).view(N, n_v).float()
    dev = dict(dtype=torch.int32, device=cuda)
    u = torch.empty(N, device=cuda)
    kept, n_kept, bud = torch.empty(N, **dev), torch.empty(1, **dev), torch.empty(N, **dev)
    sel, off = torch.full((N * n_v,), -1, **dev), torch.empty(N + 1, **dev)
    riftlib.select_budgeted_tokens(r.to(cuda), torch.full((N,), 0.25, device=cuda), N, n_v, None, riftlib.make_policy(pol),
                                   u, kept, n_kept, bud, sel, off, None, 0)
    riftlib.sync_status()
    assert int(n_kept.item()) == N and bool((u == 1).all()) and bool((bud == C).all())
    assert torch.equal(kept.cpu(), torch.arange(N, dtype=torch.int32))
    assert torch.equal(off.cpu(), torch.arange(N + 1, dtype=torch.int32) * C)
    got = sel.view(-1)[:N * C].view(N, C).cpu()
    for i in (0, 1, N // 2, N - 1):
        assert got[i].tolist() == O.top_b(r[i].numpy(), C)
    assert bool((got[:, 1:] > got[:, :-1]).all())
