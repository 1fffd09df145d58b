"""A likelihood and a posterior (or path) of one sequence in turn keep both their
plans: neither builds, uploads or waits again. A caller's capture shows it, in
which a plan's upload and its wait are not allowed.
"""
import numpy as np
import pytest
import torch

from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk_len", [0, 256])
def test_calls_in_turn_inside_a_capture(cuda_lib, chunk_len):
    api = cuda_lib
    rng = np.random.default_rng(4)
    prm = synth.random_params(7, rng)
    o = synth.sample_observations(prm, 9001, rng)
    dev, xy, fl = api.to_device(prm), torch.from_numpy(o.xy).cuda(), torch.from_numpy(o.tremor).cuda()
    opt = api.make_opts(chunk_len=chunk_len)
    ctx = api.Context()

    def calls(stream=None):
        ll = ctx.hmm_loglik(*dev, xy, fl, opts=opt, stream=stream)
        g, _ = ctx.hmm_posterior(*dev, xy, fl, opts=opt, stream=stream)
        path, _, _ = ctx.hmm_viterbi(*dev, xy, fl, opts=opt, stream=stream)
        return ll, g, path, ctx.hmm_loglik(*dev, xy, fl, opts=opt, stream=stream)

    try:
        want = [t.clone() for t in calls()]
        want = [t.clone() for t in calls()]
        torch.cuda.synchronize()
        s, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s, capture_error_mode="relaxed"):
            got = calls(s)
        graph.replay()
        torch.cuda.synchronize()
        for a, b in zip(got, want):
            assert torch.equal(a, b)
        assert ctx.hmm_status() == api.HMM_OK
    finally:
        ctx.close()
