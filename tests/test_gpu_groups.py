"""The filtered assignment and the merge of large groups, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from oracle import parity
import paper_2609_36835_gb300 as pk
from paper_2609_36835_gb300 import workload

pytestmark = pytest.mark.gpu
TAU = 1e-4   # similarity gap inside which the assignment may differ, as in the other parity tests


@pytest.fixture(scope="module", autouse=True)
def _gpu(lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _layer(H, T, n_pos, t, **kw):
    w = synth.WORKLOADS["llama8b_layer_T8192"]
    arr = workload.layer_inputs_np(w, 0, list(range(H)), T=T, n_pos=n_pos)
    return arr, workload.to_device(arr, "cuda"), workload.layer_config(w, H, T=T, n_pos=n_pos, t=t, **kw)


def _logits(arr, h):
    K, Q = synth.bf16_to_f64(arr["K"][h]), synth.bf16_to_f64(arr["Q"][h])
    return K, oracle.attention_logits(Q, K, 1.0 / np.sqrt(128.0))


# around the rule's edge (t = 23 tiles of 128 anchors, 4096 other keys): just below it
# (the full GEMM), just above it with one anchor in the last tile, odd T, a key chunk's
# ragged end, a ragged and a one-slab reduction
@pytest.mark.parametrize("H,T,n_pos,t", [(1, 7041, 10, 2944), (1, 7041, 10, 2945), (2, 9001, 16, 3001),
                                         (1, 12300, 33, 3200), (1, 7200, 260, 2950)])
def test_filtered_assignment_is_the_argmax(H, T, n_pos, t):
    arr, ten, cfg = _layer(H, T, n_pos, t)
    rng = np.random.default_rng(t)
    S = np.stack([np.sort(rng.permutation(T)[:t]) for _ in range(H)])
    out = pk.compact_layer(cfg, ten["K"], ten["V"], ten["Q"], None, None, want_assign=True,
                           anchors_in=torch.as_tensor(S, dtype=torch.int32, device="cuda"))
    for h in range(H):
        _, l = _logits(arr, h)
        u, _ = oracle.response_profiles(l)
        ok, n_mis, n_tie, worst = parity.assignment_valid_profiles(out["assign"][h].cpu().numpy(), u, S[h], TAU)
        assert ok, (h, n_mis, n_tie, worst)


# groups of 1, 128, 129, 512 + 1 and what is left of T: both counting sorts (T = 2048 and
# above), the warp's and the CTAs' merge and their remainders.  Weights carry the fp32
# error of log phi (|log phi| < 128: 8e-6), C_k with it: 2e-5.
@pytest.mark.parametrize("T", [1500, 2048, 5003])
def test_merge_of_large_groups(T):
    H, t = 2, 6
    arr, ten, cfg = _layer(H, T, 40, t, lambda_m=1.0)
    sizes = [1, 128, 129, 513, 2]
    kappa = np.repeat(np.arange(t), sizes + [T - sum(sizes)])
    S = np.concatenate([[0], np.cumsum(sizes)])
    perm = np.random.default_rng(T).permutation(T)      # the groups' members lie anywhere
    kap = np.empty(T, dtype=np.int64)
    kap[perm] = kappa
    order = np.argsort(perm[S])                          # anchors ascending; group r is the r-th anchor's
    anchors, rank = perm[S][order], np.empty(t, dtype=np.int64)
    rank[order] = np.arange(t)
    kap = rank[kap]
    A = torch.as_tensor(np.stack([anchors] * H), dtype=torch.int32, device="cuda")
    G = torch.as_tensor(np.stack([kap] * H), dtype=torch.int32, device="cuda")
    out = pk.compact_layer(cfg, ten["K"], ten["V"], ten["Q"], None, None, anchors_in=A, assign_in=G)
    for h in range(H):
        K, l = _logits(arr, h)
        C_k, _ = oracle.merge_keys(K, kap, oracle.log_mass_weights(l), anchors, 1.0)
        assert parity.rel_fro(out["C_k"][h].cpu().numpy(), C_k) <= 2e-5, h
