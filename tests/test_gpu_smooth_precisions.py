"""Posterior rows, E-step statistics, gradient and EM step with opts.precision
other than FP32: where strands carry the sequence, every vector is FP32, so the
results are those of the FP32 call, and meet its bar, whatever the precision
(gamma 8e-5: test_gpu_smooth.py; the statistics 1e-5 of the largest entry of
their kind: test_gpu_stats.py). A sequence left to the chunk products (rare tremors:
its vectors meet too late) carries their operands' rounding at chunk boundaries,
whose size depends on the chain; it has the bits of the call with the vectors off.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["tf32", "tf32_split", "bf16"])
@pytest.mark.parametrize("K,sparse", [(12, True), (32, False), (32, True), (40, False)])
def test_every_precision_smooths_in_fp32(cuda_lib, K, sparse, prec):
    api = cuda_lib
    rng = np.random.default_rng(1500 + K)
    prm = synth.random_params(K, rng, **({"p_range": synth.SPARSE_P_RANGE} if sparse else {}))
    o = synth.sample_observations(prm, 20_000, rng)
    dev = api.to_device(prm)
    xy, fl = torch.from_numpy(o.xy).cuda(), torch.from_numpy(o.tremor).cuda()
    ctx = api.Context()
    try:
        opt, plain = api.make_opts(precision=prec), api.make_opts()
        g, ll = ctx.hmm_posterior(*dev, xy, fl, opts=opt)
        ref, rll = oracle.posterior(prm, o.xy, o.tremor)
        err = np.abs(g.cpu().numpy() - ref).max()
        if ctx.last_chunk_proposals():
            ctx.set_strands(False)
            assert sparse and torch.equal(g, ctx.hmm_posterior(*dev, xy, fl, opts=opt)[0])
            return
        assert err <= 8e-5, err
        assert abs(float(ll.item()) - rll) <= 1e-6 * abs(rll) + 1e-4
        st, _ = ctx.hmm_expected_stats(*dev, xy, fl, opts=opt)
        want, _ = oracle.expected_stats(prm, o.xy, o.tremor)
        for name in want:
            scale = np.abs(want[name]).max()
            np.testing.assert_allclose(st[name].cpu().numpy(), want[name], rtol=1e-5, atol=1e-5 * scale, err_msg=name)
        for a, b in zip(ctx.hmm_loglik_grad(*dev, xy, fl, opts=opt)[0], ctx.hmm_loglik_grad(*dev, xy, fl, opts=plain)[0]):
            assert torch.allclose(a, b, rtol=1e-5, atol=1e-5 * float(b.abs().max()))
        for a, b in zip(ctx.hmm_em_step(*dev, xy, fl, opts=opt)[0], ctx.hmm_em_step(*dev, xy, fl, opts=plain)[0]):
            assert torch.allclose(a, b, rtol=1e-5, atol=1e-5 * float(b.abs().max()))
        assert ctx.hmm_status() == api.HMM_OK
    finally:
        ctx.close()
