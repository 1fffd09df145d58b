"""Outputs at addresses that are only 4-byte aligned, as the C ABI allows for
float arrays: the posterior's rows have the same bits as at an aligned address.
"""
import ctypes

import numpy as np
import pytest
import torch

from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [4, 8, 12, 32, 64, 6])
def test_posterior_rows_at_any_float_address(cuda_lib, K):
    api = cuda_lib
    rng = np.random.default_rng(K)
    prm = synth.random_params(K, rng)
    o = synth.sample_observations(prm, 3001, rng)
    dev = api.to_device(prm)
    xy, fl = torch.from_numpy(o.xy).cuda(), torch.from_numpy(o.tremor).cuda()
    ctx = api.Context()
    try:
        want, _ = ctx.hmm_posterior(*dev, xy, fl)
        p = api.hmm_params(K, *(t.data_ptr() for t in dev))
        ob = api.hmm_obs(3001, xy.data_ptr(), fl.data_ptr())
        ll = torch.empty(1, dtype=torch.float64, device="cuda")
        for off in (1, 2, 3, 4):
            flat = torch.full((3001 * K + 8,), -1.0, dtype=torch.float32, device="cuda")
            rc = ctx.lib.hmm_posterior(ctx.h, ctypes.byref(p), ctypes.byref(ob), ctypes.byref(api.make_opts()),
                                       flat.data_ptr() + 4 * off, ll.data_ptr(), torch.cuda.current_stream().cuda_stream)
            assert rc == api.HMM_OK
            assert torch.equal(flat[off:off + 3001 * K].view(3001, K), want)
            assert bool((flat[:off] == -1).all()) and bool((flat[off + 3001 * K:] == -1).all())
        assert ctx.hmm_status() == api.HMM_OK
    finally:
        ctx.close()
