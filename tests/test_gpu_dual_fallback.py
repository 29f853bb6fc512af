"""The dual fits above the sliced products' range (more than 26214 anchors): fp64 on
SIMT tile products throughout.  The oracle's primal system would be t x t, so the
reference solves the n x n dual of the same equations in fp64,
    w = Phi^T a,  (Phi Phi^T + lam I) a = m,  lam = ridge ||Phi||^2 / t,
which it has in common with the primal; the bound is that of the other parity
tests (2e-3)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from oracle import parity
import paper_2609_36835_gb300 as pk
from paper_2609_36835_gb300 import workload

pytestmark = pytest.mark.gpu
T, SCALE = 27000, 1.0 / np.sqrt(128.0)


def _dual_ridge(A, rhs, ridge):
    lam = ridge * np.sum(A * A) / A.shape[1]
    return A.T @ np.linalg.solve(A @ A.T + lam * np.eye(A.shape[0]), rhs)


def test_reference_is_the_primal_solution():
    rng = np.random.default_rng(0)
    A, rhs = rng.standard_normal((20, 50)), rng.standard_normal((20, 3))
    lam = 1e-3 * np.sum(A * A) / 50
    assert parity.rel_fro(_dual_ridge(A, rhs, 1e-3), np.linalg.solve(A.T @ A + lam * np.eye(50), A.T @ rhs)) <= 1e-10


# just above the range: one short block, several blocks of 64 rows with a ragged last one
@pytest.mark.parametrize("H,n_pos,t", [(1, 10, 26215), (2, 50, 26300)])
def test_fits_above_the_sliced_range(lib, H, n_pos, t):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = synth.WORKLOADS["llama8b_layer_T8192"]
    arr = workload.layer_inputs_np(w, 0, list(range(H)), T=T, n_pos=n_pos)
    ten = workload.to_device(arr, "cuda")
    cfg = workload.layer_config(w, H, T=T, n_pos=n_pos, t=t)
    rng = np.random.default_rng(t)
    S = np.stack([np.sort(rng.permutation(T)[:t]) for _ in range(H)])
    kappa = np.stack([np.minimum(np.searchsorted(s, np.arange(T)), t - 1) for s in S])   # the next anchor
    out = pk.compact_layer(cfg, ten["K"], ten["V"], ten["Q"], None, None,
                           anchors_in=torch.as_tensor(S, dtype=torch.int32, device="cuda"),
                           assign_in=torch.as_tensor(kappa, dtype=torch.int32, device="cuda"))
    ocfg = oracle.OracleConfig(t=t)
    for h in range(H):
        K, V, Q = (synth.bf16_to_f64(arr[k][h]) for k in ("K", "V", "Q"))
        l = oracle.attention_logits(Q, K, SCALE)
        C_k, _ = oracle.merge_keys(K, kappa[h], oracle.log_mass_weights(l), S[h], ocfg.lambda_m)
        assert parity.rel_fro(out["C_k"][h].cpu().numpy(), C_k) <= 2e-3
        z = l.max(axis=1)
        p = np.exp(l - z[:, None])
        m = p.sum(axis=1)
        lc = oracle.attention_logits(Q, C_k, SCALE)
        w_star = np.maximum(_dual_ridge(np.exp(lc - z[:, None]), m, ocfg.ridge_w), 0.0)
        beta = np.clip(np.log(np.maximum(w_star, ocfg.eps_w)), ocfg.b_min, ocfg.b_max)
        eb, rest_ok = parity.beta_errors(out["beta"][h].cpu().numpy(), beta, w_star)
        assert eb <= 2e-3 and rest_ok, ("beta", h, eb, rest_ok)
        x = lc + beta
        P = np.exp(x - x.max(axis=1, keepdims=True))
        P /= P.sum(axis=1, keepdims=True)
        C_v = _dual_ridge(P, (p / m[:, None]) @ V, ocfg.ridge_v)
        assert parity.rel_fro(out["C_v"][h].cpu().numpy(), C_v) <= 2e-3, ("C_v", h)
