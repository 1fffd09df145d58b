"""Log L by strands (one forward vector per piece of a segment, joined where
the vectors of neighbouring pieces meet) against the FP64 oracle.

The bar is the FP32 path's: |d| <= 1e-6 |log L| + 1e-4. A strand's rounding is
that of one FP32 forward recursion, and a join adds at most its tolerance,
2^-15 per piece: with |log L| above 1 per step and pieces of at least 64 steps
that is below 5e-7 |log L|. Cases: every padded state count and its edges,
lengths around the piece and warm-up sizes, observations far from every state
(a window of steps that shrinks out of range and is repeated step by step),
chains that mix slowly (the join runs on), and batches in which some
proposals only are left to the chunk products (a zero in P, a chain that does
not mix, an impossible observation).
"""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


def _close(got, ref):
    if math.isinf(ref):
        return got == ref
    return abs(got - ref) <= 1e-6 * abs(ref) + 1e-4


def _batched(api, props, xy, fl, offs, **opt):
    ctx = api.Context()
    try:
        out = ctx.hmm_loglik_batched(*api.to_device(props), offs, torch.from_numpy(np.ascontiguousarray(xy)).cuda(),
                                     torch.from_numpy(np.ascontiguousarray(fl)).cuda(), opts=api.make_opts(**opt))
        got = out.cpu().numpy()
        return got, ctx.hmm_status()
    finally:
        ctx.close()


def _check(api, props, xy, fl, offs, status=0, **opt):
    ref = oracle.loglik_batched(props, xy, fl, np.asarray(offs, np.int64))
    got, st = _batched(api, props, xy, fl, offs, **opt)
    assert st == status
    for q in range(len(ref)):
        assert _close(got[q], ref[q]), (q, got[q], ref[q])


@pytest.mark.parametrize("K", [1, 2, 4, 5, 8, 9, 16, 17, 31, 32, 33, 48, 64, 65, 80])
@pytest.mark.parametrize("prec", ["fp32", "tf32_split"])
def test_state_counts(cuda_lib, K, prec):
    rng = np.random.default_rng(700 + K)
    gen = synth.random_params(K, rng)
    lens = [1, 2, 5, 64, 65, 127, 700, 3003]
    xy, fl, offs = synth.sample_segments(gen, lens, rng)
    props = synth.stack_params([synth.perturb_params(gen, rng) for _ in range(3)])
    if prec == "fp32":
        _check(cuda_lib, props, xy, fl, offs)
        return
    ref = oracle.loglik_batched(props, xy, fl, offs)
    got, st = _batched(cuda_lib, props, xy, fl, offs, precision=prec)
    assert st == 0
    # operands rounded to TF32: 8 sqrt(T) 2^-11 (as in test_gpu_tc.py)
    assert np.all(np.abs(got - ref) <= 8 * math.sqrt(sum(lens)) * 2.0 ** -11 + 1e-3), (got, ref)


@pytest.mark.parametrize("T", [63, 64, 65, 128, 129, 190, 193, 257, 321, 1000, 20_001])
def test_lengths(cuda_lib, T):
    rng = np.random.default_rng(T)
    gen = synth.random_params(7, rng)
    o = synth.sample_observations(gen, T, rng)
    for init_mode in (0, 1):
        ref = oracle.loglik(gen, o.xy, o.tremor, init_mode)
        got, st = _batched(cuda_lib, synth.stack_params([gen]), o.xy, o.tremor, [0, T], init_mode=init_mode)
        assert st == 0 and _close(got[0], ref), (init_mode, got, ref)


@pytest.mark.parametrize("K", [3, 12, 27, 50])
def test_far_observations(cuda_lib, K):
    """Tremors up to 700 km outside the box: steps whose best emission is
    2^-1000 and less."""
    rng = np.random.default_rng(K)
    gen = synth.random_params(K, rng)
    o = synth.sample_observations(gen, 6000, rng)
    fl, xy = o.tremor.copy(), o.xy.copy()
    at = rng.choice(6000, 60, replace=False)
    at[:2] = (0, 5999)
    fl[at] = 1
    xy[at] = rng.uniform((-700, -700), (1000, 900), (60, 2)).astype(np.float32)
    _check(cuda_lib, synth.stack_params([gen, synth.perturb_params(gen, rng)]), xy, fl, [0, 6000])


def test_slow_mixing(cuda_lib):
    """States that differ little and hours with few tremors: vectors that
    start apart need thousands of steps to meet."""
    rng = np.random.default_rng(11)
    gen = synth.random_params(6, rng, diag=(0.999, 0.9999), p_range=(0.001, 0.004))
    gen.mu[:] = (150.0, 75.0) + rng.normal(0, 2.0, (6, 2)).astype(np.float32)
    o = synth.sample_observations(gen, 60_000, rng)
    _check(cuda_lib, synth.stack_params([gen, synth.perturb_params(gen, rng)]), o.xy, o.tremor, [0, 20_000, 60_000])


@pytest.mark.parametrize("prec", ["fp32", "tf32", "tf32_split", "bf16"])
@pytest.mark.parametrize("K", [6, 20, 40])
def test_mixed_batch(cuda_lib, K, prec):
    """Proposals 1, 4 and 5 cannot be carried by strands: a zero in P, P = I,
    and a state set that cannot emit the tremors at all (zero likelihood)."""
    rng = np.random.default_rng(40 + K)
    gen = synth.random_params(K, rng)
    o = synth.sample_observations(gen, 9000, rng)
    props = [synth.perturb_params(gen, rng) for _ in range(7)]
    props[1].P[0, 1] += props[1].P[0, 2]
    props[1].P[0, 2] = 0.0
    props[4].P[:] = np.eye(K, dtype=np.float32)
    props[4].mu[:] = (150.0, 75.0)
    props[4].cov[:] = (900.0, 0.0, 900.0)
    props[4].p_tremor[:] = np.linspace(0.45, 0.55, K).astype(np.float32)
    props[5].p_tremor[:] = 0.0
    props = synth.stack_params(props)
    ref = oracle.loglik_batched(props, o.xy, o.tremor, np.array([0, 2500, 9000]))
    got, st = _batched(cuda_lib, props, o.xy, o.tremor, [0, 2500, 9000], precision=prec)
    assert st == 0 and ref[5] == -math.inf and got[5] == -math.inf
    u = {"fp32": 0.0, "tf32": 2.0 ** -11, "tf32_split": 2.0 ** -11, "bf16": 2.0 ** -8}[prec]
    tol = 8 * math.sqrt(9000) * u + (9000 * u / math.sqrt(K) if prec == "tf32" else 0) + 4 * 9000 * u * u + 1e-3
    for q in (0, 1, 2, 3, 6):
        assert abs(got[q] - ref[q]) <= max(tol, 1e-6 * abs(ref[q])), (q, got[q], ref[q])
    # P = I: the product's rows round independently, so T u in place of sqrt(T) u
    assert abs(got[4] - ref[4]) <= 9000 * u + 1e-6 * abs(ref[4]) + 1e-3, (got[4], ref[4])
