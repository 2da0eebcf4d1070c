"""Symmetric scheme in bf16 in calls of many heads: tile counts, ragged ends and head sizes at the edges, scores far beyond the range of an
exponential and NaN in some heads among ordinary ones, and a head's output, which does not depend on how many heads the call
has.  Reference: the fp64 oracle; tolerance of the other bf16 tests, 2e-2 for outputs of size 1 plus half a bf16 step of the output where
it is larger."""
import numpy as np
import pytest
import torch

import oracle
from paper_2012_01114_b200 import binding, inputs

pytestmark = pytest.mark.gpu
TOL = 2e-2


def _x(seed, B, n, H, d, scale=None):
    v, bits = inputs.tensor(seed, 4, (B, n, H, d), 1.0, "bf16", row_scale=scale)
    return v, torch.from_numpy(np.ascontiguousarray(bits).view(np.int16)).cuda().view(torch.bfloat16)


def _check(out, ref, tol=TOL):
    got = out.float().cpu().numpy().astype(np.float64)
    assert np.isfinite(got).all()
    excess = np.abs(got - ref) - 2.0 ** -8 * np.abs(ref)
    assert excess.max() <= tol, excess.max()


def _census(B, H, n, d):
    st, got = binding.psa_last_issued()
    assert st == binding.OK and got == binding.psa_skip_count(B, H, n, 0, d, binding.SYMMETRIC, binding.BF16)


@pytest.mark.parametrize("H,n,d", [(1, 257, 8), (2, 384, 128), (1, 385, 64), (3, 383, 40), (1, 513, 120), (5, 640, 64), (1, 1153, 72), (1, 2100, 16)])
def test_tile_edges(H, n, d):
    # 296 heads, two for a CTA each on 148 SMs: copies, which must be alike
    B = 296 // H
    v, x = _x(n + d, 1, n, H, d)
    out = binding.psa_attention_core(x.repeat(B, 1, 1, 1), None, None, binding.SYMMETRIC)
    _census(B, H, n, d)
    ref, _ = oracle.attention_core(v, v, v, oracle.SYMMETRIC)
    _check(out[:1], ref)
    assert (out == out[:1]).all()


def test_more_heads_than_work_at_once():
    v, x = _x(3, 1, 290, 150, 16)
    out = binding.psa_attention_core(x.repeat(4, 1, 1, 1), None, None, binding.SYMMETRIC)
    _census(4, 150, 290, 16)
    ref, _ = oracle.attention_core(v, v, v, oracle.SYMMETRIC)
    _check(out[:1], ref)
    for i in range(1, 4):
        assert torch.equal(out[i], out[0])


@pytest.mark.parametrize("n,d", [(384, 64), (300, 128), (1024, 32)])
def test_large_scores_in_some_heads(n, d):
    # rows of head 1 grow to 12 x: the weight of their own score is beyond 2^100; head 2 is scaled as a whole; 0 and 3 stay
    B, H = 25, 4
    v, _ = _x(5, 1, n, H, d)
    v[:, n // 2:, 1] *= 12.0
    v[:, :, 2] *= 8.0
    x = torch.from_numpy(v).cuda().bfloat16()
    v = x.double().cpu().numpy()
    out = binding.psa_attention_core(x.repeat(B, 1, 1, 1), None, None, binding.SYMMETRIC)
    _census(B, H, n, d)
    ref, _ = oracle.attention_core(v, v, v, oracle.SYMMETRIC)
    # outputs of head 1 reach 12 times the size, of head 2 8 times; the others keep the plain bound
    y, r = out[0].view(n, H, d), ref.reshape(n, H, d)
    for h, size in enumerate((1.0, 12.0, 8.0, 1.0)):
        _check(y[:, h], r[:, h], TOL * size)
    assert binding.psa_last_rescales() > 0 and (out == out[:1]).all()


def test_nan_stays_in_its_head():
    B, H, n, d = 40, 3, 400, 64
    v, x = _x(7, 1, n, H, d)
    x = x.repeat(B, 1, 1, 1)
    x[:, 300, 1, 5] = float("nan")
    out = binding.psa_attention_core(x, None, None, binding.SYMMETRIC).view(B, n, H, d)
    st, _ = binding.psa_last_issued()
    assert st == binding.OK and torch.isnan(out[:, :, 1]).all() and torch.isfinite(out[:, :, ::2]).all()
    v0 = np.ascontiguousarray(v[:, :, ::2])
    ref, _ = oracle.attention_core(v0, v0, v0, oracle.SYMMETRIC)
    _check(out[:1, :, ::2].reshape(1, n, -1), ref)


@pytest.mark.parametrize("n,d", [(1024, 128), (384, 64), (1153, 40)])
def test_output_does_not_depend_on_the_number_of_heads(n, d):
    # the scores of a pair are handed on in fp32 and every row has its own maximum, so a head is computed alike in any company: bit by bit
    _, x = _x(n, 1, n, 4, d)
    few = binding.psa_attention_core(x, None, None, binding.SYMMETRIC)
    many = binding.psa_attention_core(x.repeat(74, 1, 1, 1), None, None, binding.SYMMETRIC)
    assert (many == few).all()
