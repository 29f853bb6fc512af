"""Index scores at the edges of the index GEMM's tile rule: keys that fill one
128-wide tile or less stay in it however many rows there are (20 heads x 8 row
tiles are more than the SMs), one key more takes 256-wide tiles.  Against the
oracle with the bound of the other parity tests (1e-3)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from oracle import parity
import paper_2609_36835_gb300 as pk
from paper_2609_36835_gb300 import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [100, 128, 129])
def test_index_scores_at_one_key_tile(lib, T):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w, H, n_pos, t = synth.WORKLOADS["llama8b_layer_T8192"], 20, 256, 10
    arr = workload.layer_inputs_np(w, 0, list(range(H)), T=T, n_pos=n_pos)
    ten = workload.to_device(arr, "cuda")
    cfg = workload.layer_config(w, H, T=T, n_pos=n_pos, t=t)
    out = pk.compact_layer(cfg, ten["K"], ten["V"], ten["Q"], ten["X"], workload.indexer_dict(ten), want_scores=True)
    for h in (0, H - 1):
        f64 = lambda k: synth.bf16_to_f64(arr[k][h])
        W = {f: f64(f) for f in pk.INDEXER_FIELDS}
        X = np.repeat(synth.bf16_to_f64(arr["X"]), cfg.G, axis=0)
        ref = oracle.compact_pair(f64("K"), f64("V"), f64("Q"), X, W, oracle.OracleConfig(t=t), H_I=cfg.H_I)
        e_inf, e_top = parity.score_errors(out["scores"][h].cpu().numpy().astype(np.float64), ref["scores"], t)
        assert e_inf <= 1e-3 and e_top <= 1e-3, (h, e_inf, e_top)
