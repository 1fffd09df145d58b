"""The chunk products, which take what the vectors do not: their tests of sizes,
chunk lengths, renormalisation intervals, run lengths, posteriors, statistics
and paths with the vectors switched off (hmm_set_strands), at the bars of those
tests; and batches in which some proposals only are listed for them (a zero in
P), whose results have the bits of the same call with the vectors off.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2003_03508_gb300 import synth

from . import test_gpu_loglik as loglik
from . import test_gpu_posterior as posterior
from . import test_gpu_runlen as runlen
from . import test_gpu_stats as stats
from . import test_gpu_tc as tc
from . import test_gpu_viterbi as viterbi

pytestmark = pytest.mark.gpu
SIZES = [1, 4, 16, 17, 25, 32, 33, 48, 49, 64, 65, 80]


@pytest.fixture()
def chunks(cuda_lib):
    """The binding with the default context's vectors off; its last call must have taken chunk products."""
    ctx = cuda_lib.default_context()
    ctx.set_strands(False)
    try:
        yield cuda_lib
        assert ctx.last_chunk_proposals() >= 1
        assert ctx.hmm_status() == cuda_lib.HMM_OK
    finally:
        ctx.set_strands(True)


@pytest.mark.parametrize("K", SIZES)
def test_fp32_sizes(chunks, K):
    loglik.test_fp32_parity_sizes(chunks, K)


@pytest.mark.parametrize("prec", tc.PRECS)
@pytest.mark.parametrize("K", SIZES)
def test_tensor_core_sizes(chunks, K, prec):
    tc.test_tc_parity_sizes(chunks, K, prec)


@pytest.mark.parametrize("T", [2, 65, 130])
@pytest.mark.parametrize("prec", tc.PRECS)
def test_tensor_core_lengths(chunks, T, prec):
    tc.test_tc_small_T(chunks, prec, T)
    for K in (64, 80):
        tc.test_tc_wide_small_T(chunks, prec, K, T)


@pytest.mark.parametrize("R", [1, 3, 8])
@pytest.mark.parametrize("prec", tc.PRECS)
def test_renorm_intervals(chunks, R, prec):
    for K in (16, 32):
        tc.test_tc_renorm_intervals(chunks, prec, K, R)


def test_fp32_renorm_intervals(chunks):
    loglik.test_renorm_interval_invariance(chunks)


@pytest.mark.parametrize("prec", tc.PRECS)
@pytest.mark.parametrize("K", [32, 48, 64, 80])
def test_segments(chunks, K, prec):
    tc.test_tc_batched_segments(chunks, prec, K)


@pytest.mark.parametrize("K", [1, 2, 3, 7, 16, 25, 32, 33, 48, 64, 80])
def test_run_lengths(chunks, K):
    runlen.test_parity_sizes(chunks, K)


def test_run_length_segments(chunks):
    runlen.test_batched_ragged_segments(chunks)


@pytest.mark.parametrize("K", [2, 3, 7, 16, 25, 32, 33, 64, 80])
def test_posterior_sizes(chunks, K):
    posterior.test_posterior_parity_sizes(chunks, K)


@pytest.mark.parametrize("prec,tol", [("tf32", 1e-3), ("tf32_split", 1e-3), ("bf16", 2e-2)])
def test_posterior_from_tensor_core_products(chunks, prec, tol):
    posterior.test_posterior_tensor_core_products(chunks, prec, tol)


@pytest.mark.parametrize("K", [2, 3, 16, 25, 32, 64])
def test_statistics_sizes(chunks, K):
    stats.test_stats_parity(chunks, K)


@pytest.mark.parametrize("K", [2, 3, 7, 16, 25, 32, 33, 64, 80])
def test_path_sizes(chunks, K):
    viterbi.test_viterbi_parity_sizes(chunks, K)


@pytest.mark.parametrize("prec,run", [("fp32", 0), ("fp32", 4), ("tf32", 0), ("tf32_split", 0), ("bf16", 0)])
@pytest.mark.parametrize("K", [4, 8, 16, 32, 48, 60, 80])
def test_listed_proposals(cuda_lib, K, prec, run):
    """Proposals 1, 2 and 6 of 7 have a zero in P."""
    api = cuda_lib
    rng = np.random.default_rng(90 + K)
    gen = synth.random_params(K, rng, **({"p_range": synth.SPARSE_P_RANGE} if run else {}))
    o = synth.sample_observations(gen, 7000, rng)
    props = [synth.perturb_params(gen, rng) for _ in range(7)]
    for q in (1, 2, 6):
        props[q].P[0, 1] += props[q].P[0, 2]
        props[q].P[0, 2] = 0.0
    props = synth.stack_params(props)
    offs = np.array([0, 2500, 7000], np.int64)
    ref = oracle.loglik_batched(props, o.xy, o.tremor, offs)
    dev, xy, fl = api.to_device(props), torch.from_numpy(o.xy).cuda(), torch.from_numpy(o.tremor).cuda()
    opt = api.make_opts(precision=prec, runlen_min=run)
    ctx = api.Context()
    try:
        got = ctx.hmm_loglik_batched(*dev, offs, xy, fl, opts=opt).cpu().numpy()
        # (FP32 beyond 64 states has chunk products alone)
        assert ctx.last_chunk_proposals() == (7 if prec == "fp32" and K > 64 else 3)
        ctx.set_strands(False)
        alone = ctx.hmm_loglik_batched(*dev, offs, xy, fl, opts=opt).cpu().numpy()
        assert ctx.last_chunk_proposals() == 7
        assert ctx.hmm_status() == api.HMM_OK
    finally:
        ctx.close()
    assert np.array_equal(got[[1, 2, 6]], alone[[1, 2, 6]])
    for v in (got, alone):
        if prec == "fp32":
            assert np.all(np.abs(v - ref) <= 1e-6 * np.abs(ref) + 1e-4), v - ref
        else:
            assert np.all(np.abs(v - ref) <= tc.tol(prec, 2500, K) + tc.tol(prec, 4500, K)), v - ref


@pytest.mark.parametrize("prec", tc.PRECS)
@pytest.mark.parametrize("K", [20, 40, 72])
def test_late_meetings_on_the_tensor_cores(cuda_lib, K, prec):
    """Rare tremors, and states that differ little: the first look fails at many
    boundaries, the join runs on in FP32 (or gives a proposal up). The reference
    has P as the precision holds it, rounded to TF32 for "tf32": with states that
    keep to themselves that rounding alone moves log L by T u and more (3.6 nats
    at K=72, by the oracle), which says nothing of the vectors. What is left is
    bounded by 8 sqrt(T) u (+ BF16's drift) as in test_gpu_tc.py."""
    api = cuda_lib
    for seed, kw in ((1, {"p_range": synth.SPARSE_P_RANGE}), (2, {"diag": (0.999, 0.9999), "p_range": (0.02, 0.2)})):
        rng = np.random.default_rng(seed + K)
        gen = synth.random_params(K, rng, **kw)
        if seed == 2:
            gen.mu[:] = (150.0, 75.0) + rng.normal(0, 2.0, (K, 2)).astype(np.float32)
        o = synth.sample_observations(gen, 40_000, rng)
        props = synth.stack_params([synth.perturb_params(gen, rng) for _ in range(64)])
        ctx = api.Context()
        try:
            got = ctx.hmm_loglik_batched(*api.to_device(props), [0, 40_000], torch.from_numpy(o.xy).cuda(),
                                         torch.from_numpy(o.tremor).cuda(), opts=api.make_opts(precision=prec)).cpu().numpy()
            print(K, prec, seed, "left to chunk products:", ctx.last_chunk_proposals())
            assert ctx.hmm_status() == api.HMM_OK
        finally:
            ctx.close()
        pick = [0, 31, 63]
        sub = type(props)(*(a[pick].copy() for a in props.as_tuple()))
        if prec == "tf32":
            bits = sub.P.view(np.uint32)
            sub.P[:] = ((bits + np.uint32(0x1000)) & np.uint32(0xFFFFE000)).view(np.float32)
        ref = oracle.loglik_batched(sub, o.xy, o.tremor, np.array([0, 40_000]), n_threads=3)
        bar = tc.tol("tf32_split" if prec == "tf32" else prec, 40_000, K)
        assert np.all(np.abs(got[pick] - ref) <= bar), got[pick] - ref
