"""The number of kernels that a call reports, against the launch sequence: an
assignment of its own in place of a given one changes only that stage, whose
launches are known (given: log phi and the two checks)."""
import numpy as np
import pytest
import torch

import synth
import paper_2609_36835_gb300 as pk
from paper_2609_36835_gb300 import workload

pytestmark = pytest.mark.gpu
GIVEN = 3


@pytest.fixture(scope="module", autouse=True)
def _gpu(lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


# keys that are not anchors: column profiles, one product, the decoding; none: no product
@pytest.mark.parametrize("T,t,stage", [(600, 50, 3), (603, 50, 3), (60, 60, 2)])
def test_assignment_launches(T, t, stage):
    w = synth.WORKLOADS["llama8b_layer_T8192"]
    ten = workload.to_device(workload.layer_inputs_np(w, 0, [0], T=T, n_pos=20), "cuda")
    cfg = workload.layer_config(w, 1, T=T, n_pos=20, t=t)
    S = torch.as_tensor(np.sort(np.random.default_rng(t).permutation(T)[:t])[None], dtype=torch.int32, device="cuda")
    call = lambda **kw: pk.compact_layer(cfg, ten["K"], ten["V"], ten["Q"], None, None, anchors_in=S, want_assign=True, **kw)
    own = call()
    assert own["launches"] - call(assign_in=own["assign"])["launches"] == stage - GIVEN
