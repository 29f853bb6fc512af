"""Fits of values near the end of fp32's range.  C_v is linear in V, and scaling by
a power of two is exact, so the fit of V 2^-112 is 2^-112 times the fit of V up to
what subnormal numbers round: 2^-149 absolute, 2^-33 of a right-hand side of 2^-116,
times the system's condition t / ridge_v = 2^18: 3e-5, bound 1e-4."""
import numpy as np
import pytest
import torch

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


# several 64-wide blocks of the primal solver: trailing updates and back substitution
@pytest.mark.parametrize("T,n_pos,t", [(400, 90, 257), (900, 161, 577)])
def test_values_near_the_subnormal_range(T, n_pos, t):
    w = synth.WORKLOADS["llama8b_layer_T8192"]
    ten = workload.to_device(workload.layer_inputs_np(w, 0, [0], T=T, n_pos=n_pos), "cuda")
    cfg = workload.layer_config(w, 1, T=T, n_pos=n_pos, t=t)
    S = np.sort(np.random.default_rng(t).permutation(T)[:t])
    kappa = np.abs(np.arange(T)[:, None] - S[None, :]).argmin(axis=1)   # the nearest anchor
    given = dict(anchors_in=torch.as_tensor(S[None], dtype=torch.int32, device="cuda"),
                 assign_in=torch.as_tensor(kappa[None], dtype=torch.int32, device="cuda"))
    fit = lambda V: pk.compact_layer(cfg, ten["K"], V, ten["Q"], None, None, **given)["C_v"].cpu().numpy().astype(np.float64)
    ref = fit(ten["V"])
    small = fit(ten["V"] * 2.0 ** -112) * 2.0 ** 112
    assert parity.rel_fro(small, ref) <= 1e-4
