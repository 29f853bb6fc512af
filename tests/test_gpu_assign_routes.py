"""The assignment's routes against one another: the filter and its second pass
compare the scores of the full product, so both give the same groups whatever the
data.  With the caller's anchors H_I only sizes the workspace: with one index head
its halves do not hold the filter's lists, and the full product is the only route."""
import numpy as np
import pytest
import torch

import paper_2609_36835_gb300 as pk

pytestmark = pytest.mark.gpu
D = 128
GIVEN, FULL, FILTERED = 3, 3, 9   # launches of the stage (given: log phi and the two checks)


@pytest.fixture(scope="module", autouse=True)
def _gpu(lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _share(K, Q, S):
    """The share of (key, 128 anchors) pairs that the filter's bounds leave open, over 256 keys."""
    def profiles(k):
        l = Q.float() @ k.float().T / D ** 0.5
        e = torch.exp(l - l.amax(dim=0))
        return e / e.norm(dim=0)
    u, a = profiles(K[:: K.shape[0] // 256][:256]), profiles(K[S.long()])
    h, g = u.bfloat16().float(), a.bfloat16().float()
    ru, ra = (u - h).norm(dim=0), (a - g).norm(dim=0)
    x = h.T @ g
    line = (x - ra).amax(dim=1) - 2 * (ru + 2.0 ** -15 + Q.shape[0] * 2.0 ** -22)
    return (torch.stack([c.amax(dim=1) for c in (x + ra).split(128, dim=1)], dim=1) >= line[:, None]).float().mean().item()


# (H, T, n_pos, t, kind): the largest reduction, short key chunks; a ragged chunk, one
# anchor in the last tile, odd T; a ragged reduction and sample step; every key alike, half
# of them alike (the sample's other answer); sizes at which the filter is not tried
@pytest.mark.parametrize("H,T,n_pos,t,kind,tried", [
    (1, 20000, 512, 8000, "far", True), (2, 30001, 128, 5889, "far", True), (1, 26003, 253, 5201, "near", True),
    (1, 27500, 128, 5300, "same", True), (2, 27500, 129, 5300, "half", True),
    (1, 9500, 127, 4400, "far", False), (1, 9500, 128, 4200, "far", False)])
def test_routes_agree(H, T, n_pos, t, kind, tried):
    g = torch.Generator(device="cuda").manual_seed(T + t)
    draw = lambda *s: torch.randn(*s, device="cuda", generator=g)
    # "far": keys in 200 well separated directions, "near": unit keys
    K = draw(H, T, D)
    if kind == "far":
        c = 6 * draw(H, 200, D)
        K = K * 0.7 + torch.gather(c, 1, (torch.arange(T, device="cuda") * 200 // T)[None, :, None].expand(H, -1, D))
    if kind in ("same", "half"):
        K[:, : T if kind == "same" else T // 2] = K[:, :1]
    K, V, n = K.bfloat16(), draw(H, T, D).bfloat16(), 4 * n_pos
    pick = torch.randint(T, (H, n), device="cuda", generator=g)
    Q = (torch.gather(K, 1, pick[..., None].expand(-1, -1, D)).float() + 0.5 * draw(H, n, D)).bfloat16()
    S = torch.stack([torch.randperm(T, device="cuda", generator=g)[:t].sort().values for _ in range(H)]).int()
    out = {}
    for H_I in (8, 1):
        cfg = pk.Config(H_kv=H, T=T, n_pos=n_pos, t=t, d_x=4096, H_I=H_I)
        call = lambda **kw: pk.compact_layer(cfg, K, V, Q, None, None, anchors_in=S, want_assign=True, **kw)
        o = call()
        out[H_I] = o["assign"]
        stage = o["launches"] - call(assign_in=o["assign"])["launches"] + GIVEN
        assert stage == (FILTERED if tried and H_I == 8 else FULL), (H_I, stage)
    assert torch.equal(out[8], out[1])
    if kind == "far" and tried:   # well below the sample's line: the filter's own passes gave out[8]
        assert max(_share(K[h], Q[h], S[h]) for h in range(H)) < 0.2
    if kind == "same":
        assert min(_share(K[h], Q[h], S[h]) for h in range(H)) == 1.0
