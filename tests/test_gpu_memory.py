"""A batch whose chunk products just fit the device's memory is evaluated with
them; the vectors' workspace beside them is not asked for at any price.

2048 proposals of four states on 4096 segments of 65 observations: chunk products
0.67 GB (0.75 with what a context reserves beyond), vectors 0.44 GB more. The device
is filled up to 1 GB by a tensor that is never touched.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


def test_chunk_products_where_vectors_do_not_fit(cuda_lib):
    api = cuda_lib
    K, n, segs = 4, 2048, 4096
    rng = np.random.default_rng(1)
    gen = synth.random_params(K, rng)
    o = synth.sample_observations(gen, 65 * segs, rng)
    offs = np.arange(0, 65 * segs + 1, 65, dtype=np.int64)
    few = [synth.perturb_params(gen, rng) for _ in range(4)]
    dev = api.to_device(synth.stack_params(few * (n // 4)))
    xy, fl = torch.from_numpy(o.xy).cuda(), torch.from_numpy(o.tremor).cuda()
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    warm = api.Context()
    small = np.array([0, 65], np.int64)
    for on in (True, False):  # the kernels are loaded before memory is short
        warm.set_strands(on)
        warm.hmm_loglik_batched(*dev, small, xy, fl, out=out)
    torch.cuda.synchronize()
    warm.close()
    ctx, hold = api.Context(), None
    try:
        torch.cuda.empty_cache()
        hold = torch.empty(torch.cuda.mem_get_info()[0] - (1000 << 20), dtype=torch.uint8, device="cuda")
        for _ in range(3):
            ctx.hmm_loglik_batched(*dev, offs, xy, fl, out=out)
            assert ctx.last_chunk_proposals() == n
        tight = out.cpu().numpy().copy()
        assert ctx.hmm_status() == api.HMM_OK
        del hold
        hold = None
        torch.cuda.empty_cache()
        ctx.set_strands(True)
        ctx.hmm_loglik_batched(*dev, offs, xy, fl, out=out)
        assert ctx.last_chunk_proposals() == 0
        roomy = out.cpu().numpy()
    finally:
        del hold
        ctx.close()
        torch.cuda.empty_cache()
    ref = oracle.loglik_batched(synth.stack_params(few), o.xy, o.tremor, offs, n_threads=4)
    for got in (tight, roomy):
        assert np.all(np.abs(got.reshape(-1, 4) - ref) <= 1e-6 * np.abs(ref) + 1e-4)
