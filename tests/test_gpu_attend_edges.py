"""Joint and compact attention and the truncated-output error at the edges of
their tiles (16 keys a warp, four warps; 32 or 64 rows, 64 keys): every head against the oracle,
with the bound of the other joint-attention tests (1e-4)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_36835_gb300 as pk

pytestmark = pytest.mark.gpu
SCALE = 1.0 / np.sqrt(128.0)


@pytest.fixture(scope="module", autouse=True)
def _gpu(lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _draw(seed, *shape, dtype=torch.bfloat16):
    g = torch.Generator().manual_seed(seed)
    return torch.randn(*shape, generator=g).to(dtype)


def _np(x):
    return x.double().numpy()


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


# (H, n, t, F, compact type): one key of each block, a tile's and a round's edge,
# a block boundary inside a warp's round, one split and many, ragged query rows
@pytest.mark.parametrize("H,n,t,F,dtype", [
    (1, 1, 1, 1, torch.float32), (2, 4, 16, 0, torch.float32), (2, 5, 17, 47, torch.bfloat16),
    (3, 4, 64, 1, torch.float32), (2, 3, 65, 63, torch.bfloat16), (700, 4, 0, 65, torch.bfloat16),
    (8, 8, 333, 4001, torch.float32)])
def test_joint_tile_edges(H, n, t, F, dtype):
    Q, Kf, Vf = _draw(1, H, n, 128) * 2, _draw(2, H, F, 128), _draw(3, H, F, 128)
    Ck, Cv, beta = _draw(4, H, t, 128, dtype=dtype), _draw(5, H, t, 128, dtype=dtype), _draw(6, H, t, dtype=torch.float32)
    if t > 32:
        beta[:, 8:29] = -float("inf")   # a masked stretch longer than a tile: weight exactly 0
    dev = lambda x, on: x.cuda() if on else None
    O = pk.attend_joint(Q.cuda(), dev(Ck, t), dev(beta, t), dev(Cv, t), dev(Kf, F), dev(Vf, F)).cpu().numpy()
    for h in range(H):
        x = np.concatenate([_np(Q[h]) @ _np(Ck[h]).T * SCALE + _np(beta[h]), _np(Q[h]) @ _np(Kf[h]).T * SCALE], axis=1)
        p = np.exp(x - x.max(axis=1, keepdims=True))
        ref = p / p.sum(axis=1, keepdims=True) @ np.concatenate([_np(Cv[h]), _np(Vf[h])])
        assert _rel(O[h], ref) <= 1e-4, h


# (H, n, t): 32-row tiles with key splits, 64-row tiles, odd pitches, a slab's edge, one key
@pytest.mark.parametrize("H,n,t", [(1, 1, 1), (2, 33, 63), (1, 70, 1027), (8, 900, 65), (3, 5, 4097)])
def test_compact_attention_tile_edges(H, n, t):
    Q, Ck, Cv = _draw(1, H, n, 128) * 2, _draw(4, H, t, 128, dtype=torch.float32), _draw(5, H, t, 128, dtype=torch.float32)
    beta = _draw(6, H, t, dtype=torch.float32)
    beta[:, 1::3] = -20.0
    O = pk.attend(Q.cuda(), Ck.cuda(), beta.cuda(), Cv.cuda()).cpu().numpy()
    for h in range(H):
        ref = oracle.compact_attention(_np(Q[h]), _np(Ck[h]), _np(beta[h]), _np(Cv[h]), SCALE)
        assert _rel(O[h], ref) <= 1e-4, h


@pytest.mark.parametrize("H,n,T,t", [(1, 1, 2, 1), (2, 5, 17, 3), (3, 6, 1030, 100), (8, 16, 3001, 3000)])
def test_truncated_error_tile_edges(H, n, T, t):
    Q, K, V = _draw(7, H, n, 128), _draw(8, H, T, 128), _draw(9, H, T, 128)
    g = torch.Generator().manual_seed(10)
    S = torch.stack([torch.randperm(T, generator=g)[:t].sort().values for _ in range(H)]).int()
    E = pk.truncated_error(Q.cuda(), K.cuda(), V.cuda(), S.cuda()).cpu().numpy()
    for h in range(H):
        ref = oracle.truncated_output_error(_np(Q[h]), _np(K[h]), _np(V[h]), S[h].numpy(), SCALE)
        assert abs(E[h] - ref) <= 1e-4 * max(ref, 1e-2), (h, E[h], ref)
