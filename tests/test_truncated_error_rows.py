"""E(S) over many query rows: where the rows alone fill the GPU the keys are not
split, and a row costs its error of four bytes, not the partial outputs of a split."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_36835_gb300 as pk


# split and unsplit keys, the most query rows that a call takes
@pytest.mark.parametrize("H,n", [(8, 64), (64, 131072), (1, 262140)])
def test_workspace_does_not_hold_unsplit_rows(lib, H, n):
    T, t = 4096, 64
    need = lib.arckv_truncated_error_workspace_bytes(H, n, T, t, 128)
    # the mask, four bytes a row, and at most 32 MB of splits' partial rows (1 KB each)
    assert 0 < need <= H * T + 4 * H * n + (32 << 20)


# 2,800 blocks of four rows, the last of one row: one split; a tile's edge
@pytest.mark.gpu
@pytest.mark.parametrize("T,t", [(1, 0), (70, 11), (257, 257)])
def test_rows_of_one_split(lib, T, t):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    H, n = 700, 13
    g = torch.Generator().manual_seed(T)
    Q, K, V = (torch.randn(H, m, 128, generator=g).bfloat16() for m in (n, T, T))
    S = torch.stack([torch.randperm(T, generator=g)[:t].sort().values for _ in range(H)]).int()
    E = pk.truncated_error(Q.cuda(), K.cuda(), V.cuda(), S.cuda() if t else None).cpu().numpy()
    for h in range(0, H, 7):
        ref = oracle.truncated_output_error(Q[h].double().numpy(), K[h].double().numpy(), V[h].double().numpy(),
                                            S[h].numpy(), 1.0 / np.sqrt(128.0))
        assert abs(E[h] - ref) <= 1e-4 * max(ref, 1e-2), (h, E[h], ref)
