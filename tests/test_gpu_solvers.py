"""The primal fits' solvers at the edges of their block and cluster sizes:
merge and fits on given anchors and groups, every head against the oracle's
closed forms, with the bound of the other parity tests (2e-3)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from oracle import parity
import paper_2609_36835_gb300 as pk
from paper_2609_36835_gb300 import workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu(lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


# one block (full, short, one row), its edge, the cluster sizes 4 / 8 / 12 or 16
# (5 and 9 blocks; 8 heads at a time), and one above the clustered substitution's 2048
@pytest.mark.parametrize("H,T,n_pos,t", [(2, 200, 40, 1), (2, 200, 40, 64), (2, 203, 40, 65), (1, 400, 90, 257),
                                         (3, 801, 160, 513), (8, 900, 161, 577), (1, 2500, 600, 2049),
                                         # reference attention: 64-row tiles (split and odd T), 32-row tiles at odd T
                                         (8, 704, 128, 70), (4, 705, 290, 60), (8, 701, 128, 70)])
def test_primal_fits_on_given_groups(H, T, n_pos, t):
    w = synth.WORKLOADS["llama8b_layer_T8192"]
    arr = workload.layer_inputs_np(w, 0, list(range(H)), T=T, n_pos=n_pos)
    ten = workload.to_device(arr, "cuda")
    cfg = workload.layer_config(w, H, T=T, n_pos=n_pos, t=t)
    rng = np.random.default_rng(t)
    S = np.stack([np.sort(rng.permutation(T)[:t]) for _ in range(H)])
    kappa = np.stack([np.abs(np.arange(T)[:, None] - s[None, :]).argmin(axis=1) for s in S])   # the nearest anchor
    out = pk.compact_layer(cfg, ten["K"], ten["V"], ten["Q"], None, None,
                           anchors_in=torch.as_tensor(S, dtype=torch.int32, device="cuda"),
                           assign_in=torch.as_tensor(kappa, dtype=torch.int32, device="cuda"))
    ocfg, scale = oracle.OracleConfig(t=t), 1.0 / np.sqrt(128.0)
    for h in range(H):
        K, V, Q = (synth.bf16_to_f64(arr[k][h]) for k in ("K", "V", "Q"))
        logphi = oracle.log_mass_weights(oracle.attention_logits(Q, K, scale))
        C_k, _ = oracle.merge_keys(K, kappa[h], logphi, S[h], ocfg.lambda_m)
        fb = oracle.fit_beta(Q, K, C_k, ocfg, scale)
        fv = oracle.fit_values(Q, K, V, C_k, fb["beta"], ocfg, scale)
        assert parity.rel_fro(out["C_k"][h].cpu().numpy(), C_k) <= 2e-3
        eb, rest_ok = parity.beta_errors(out["beta"][h].cpu().numpy(), fb["beta"], fb["w_star"])
        assert eb <= 2e-3 and rest_ok, ("beta", h, eb, rest_ok)
        assert parity.rel_fro(out["C_v"][h].cpu().numpy(), fv["C_v"]) <= 2e-3, ("C_v", h)
