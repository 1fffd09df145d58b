"""Chains that do not mix: what is spent on vectors that never meet is bounded by
what the chunk products of the call take. Each call with the vectors on, which
gives up, against the vectors off: half as long again by the bound, and the
vectors' own passes (a third at the sizes here). In the smallest calls the 256 to 320 steps
that every join may have are more than that bound: 0.3 ms beyond 32 states, two
thirds of the K=48 batch here. 3 is asked for; joins that ran on for a fixed
number of steps took 2.4 to 8 times as long. Results are the oracle's.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


def _chain(K, T):
    rng = np.random.default_rng(K)
    g = synth.random_params(K, rng)
    g.P[:] = 1e-6
    np.fill_diagonal(g.P, 1.0 - 1e-6 * (K - 1))
    g.mu[:] = (150.0, 75.0)
    g.cov[:] = (900.0, 0.0, 900.0)
    g.p_tremor[:] = np.linspace(0.45, 0.55, K).astype(np.float32)
    return g, synth.sample_observations(g, T, rng)


def _ms(call):
    best = float("inf")
    for _ in range(6):
        e0, e1 = torch.cuda.Event(True), torch.cuda.Event(True)
        e0.record()
        out = call()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best, out


@pytest.mark.parametrize("K,T,n,prec", [(6, 10_000, 1, "fp32"), (16, 16_384, 256, "tf32_split"), (32, 131_072, 64, "tf32"),
                                        (48, 5000, 16, "tf32"), (64, 100_000, 64, "tf32"), (80, 65_536, 32, "bf16"),
                                        (45, 9000, 20, "fp32")])
def test_batch(cuda_lib, K, T, n, prec):
    api = cuda_lib
    g, o = _chain(K, T)
    dev = api.to_device(synth.stack_params([g] * n))
    xy, fl = torch.from_numpy(o.xy).cuda(), torch.from_numpy(o.tremor).cuda()
    buf = torch.empty(n, dtype=torch.float64, device="cuda")
    ctx = api.Context()
    try:
        call = lambda: ctx.hmm_loglik_batched(*dev, [0, T], xy, fl, opts=api.make_opts(precision=prec), out=buf)  # noqa: E731
        on, got = _ms(call)
        assert ctx.last_chunk_proposals() == n
        got = got.cpu().numpy().copy()
        ctx.set_strands(False)
        off, alone = _ms(call)
        assert np.array_equal(got, alone.cpu().numpy())
    finally:
        ctx.close()
    print(K, T, n, prec, "%.3f ms, chunk products alone %.3f" % (on, off))
    assert on <= 3.0 * off, (on, off)
    if prec == "fp32":
        ref = oracle.loglik(g, o.xy, o.tremor)
        assert np.all(np.abs(got - ref) <= 1e-6 * abs(ref) + 1e-4)


@pytest.mark.parametrize("K,T", [(6, 10_000), (16, 30_000), (25, 105_000), (48, 30_000)])
def test_posterior_and_path(cuda_lib, K, T):
    api = cuda_lib
    g, o = _chain(K, T)
    dev = api.to_device(g)
    xy, fl = torch.from_numpy(o.xy).cuda(), torch.from_numpy(o.tremor).cuda()
    ctx = api.Context()
    try:
        for name in ("hmm_posterior", "hmm_viterbi"):
            call = lambda: getattr(ctx, name)(*dev, xy, fl)  # noqa: E731
            ctx.set_strands(True)
            on, _ = _ms(call)
            ctx.set_strands(False)
            off, _ = _ms(call)
            print(K, T, name, "%.3f ms, chunk products alone %.3f" % (on, off))
            assert on <= 3.0 * off, (name, on, off)
    finally:
        ctx.close()
