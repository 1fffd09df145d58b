"""The tuner measures the chunk products themselves: among candidates whose times
are far apart it stores one of the fastest, also for a batch whose proposals
vectors carry, and says what its chunk products take.
"""
import pytest
import torch

from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,K,T,n", [("tf32", 32, 1 << 17, 64), ("fp32", 16, 1 << 16, 32)])
def test_tuned_length_is_among_the_fastest(cuda_lib, prec, K, T, n):
    api = cuda_lib
    d = synth.batched_inputs(K=K, T=T, n_prop=n, seed=3)
    dev, xy, fl = api.to_device(d["params"]), torch.from_numpy(d["xy"]).cuda(), torch.from_numpy(d["tremor"]).cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ctx = api.Context()
    api.tune_clear()
    try:
        _, L, ms = ctx.hmm_autotune_batched(*dev, d["offsets"], xy, fl, opts=api.make_opts(precision=prec), reps=5)
        assert ctx.last_chunk_proposals() == 0  # the call that leaves the result is an ordinary one
        ctx.set_strands(False)
        times = {}
        for c in api.tune_candidates(prec, n, K, T - 1, sms):
            o = api.make_opts(precision=prec, chunk_len=c)
            best = float("inf")
            for _ in range(8):
                e0, e1 = torch.cuda.Event(True), torch.cuda.Event(True)
                e0.record()
                ctx.hmm_loglik_batched(*dev, d["offsets"], xy, fl, opts=o)
                e1.record()
                torch.cuda.synchronize()
                best = min(best, e0.elapsed_time(e1))
            times[c] = best
        print(prec, "tuned", L, "%.3f ms" % ms, {c: round(t, 3) for c, t in times.items()})
        # (in FP32 the candidates are within 15% of one another)
        assert prec == "fp32" or max(times.values()) >= 1.5 * min(times.values())
        assert times[L] <= 1.15 * min(times.values())
        assert 0.7 * times[L] <= ms <= 1.4 * times[L]
    finally:
        api.tune_clear()
        ctx.close()
