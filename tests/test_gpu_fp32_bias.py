"""FP32 log L has no error that repeats at every step without a tremor.

Rare tremors: nearly all steps are quiet, and |log L| is about 0.3 a step. A
state's factor 1 - p is rounded once to FP32, at most 2^-25 of it, 1.7e-8 rms,
another way in every state and proposal; half a dozen states share the steps, so
a proposal's error is about 1.7e-8 / sqrt(6) / 0.3 = 2.3e-8 of log L, and the
mean of 32 proposals a fifth of that. Its bar is 2e-8; a factor that is too
small in the mean shows in full.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [6, 15, 32, 48])
def test_mean_error_of_rare_tremors(cuda_lib, K):
    api = cuda_lib
    d = synth.batched_inputs(K=K, T=65_536, n_prop=32, seed=K, sparse=True)
    ctx = api.Context()
    try:
        got = ctx.hmm_loglik_batched(*api.to_device(d["params"]), d["offsets"], torch.from_numpy(d["xy"]).cuda(),
                                     torch.from_numpy(d["tremor"]).cuda(), opts=api.make_opts(runlen_min=4)).cpu().numpy()
        assert ctx.hmm_status() == api.HMM_OK
    finally:
        ctx.close()
    ref = oracle.loglik_batched(d["params"], d["xy"], d["tremor"], d["offsets"], n_threads=8)
    e = (got - ref) / np.abs(ref)
    print(K, "mean %.2e rms %.2e" % (e.mean(), np.sqrt((e ** 2).mean())))
    assert abs(e.mean()) <= 2e-8, e.mean()
