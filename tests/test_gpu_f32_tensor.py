"""fp32 attention on the tensor cores (FULL from 160 vectors per head on, MASKED from 257): block and tile edges, head sizes that are not a
multiple of the tile, rows on and off the diagonal tiles, and heads whose numbers its bf16 parts cannot carry.  Reference: the fp64
oracle.  Bounds: an fp32 softmax over scores of size s is off by about 2^-24 (s + 1) per weight and the weighted sum by as much
again; 4e-6 of the output's root mean square, the accuracy that the CUDA-core path shows on these inputs, four times over."""
import numpy as np
import pytest
import torch

import oracle
from paper_2012_01114_b200 import binding, inputs

pytestmark = pytest.mark.gpu


def _run(B, H, n, d, scheme, change=None):
    t = [inputs.tensor(11 * n + d, 4 + i, (B, n, H, d), 1.0, "f32")[1] for i in range(3)]
    if change:
        change(t)
    out = binding.psa_attention_core(*[torch.from_numpy(x).cuda() for x in t], scheme)
    st, got = binding.psa_last_issued()
    assert st == binding.OK and got == binding.psa_skip_count(B, H, n, 0, d, scheme, binding.F32)
    ref, _ = oracle.attention_core(*[x.astype(np.float64) for x in t], scheme)
    return out.cpu().numpy().astype(np.float64), ref


def _close(got, ref, rel=4e-6):
    assert np.isfinite(got).all()
    assert np.linalg.norm(got - ref) <= rel * np.linalg.norm(ref)
    assert np.abs(got - ref).max() <= 10 * rel * max(np.sqrt((ref ** 2).mean()), np.abs(ref).max() / 10)


@pytest.mark.parametrize("scheme", [oracle.FULL, oracle.MASKED])
@pytest.mark.parametrize("B,H,n,d", [(2, 10, 161, 64), (4, 8, 256, 8), (2, 10, 193, 128), (2, 30, 193, 128), (2, 8, 257, 72), (4, 9, 300, 40), (1, 4, 1024, 120), (1, 6, 1000, 16), (3, 4, 513, 64), (1, 9, 705, 128),
                                     (2, 20, 384, 8), (2, 32, 257, 64), (1, 41, 257, 128), (3, 13, 300, 48), (1, 24, 385, 32), (7, 3, 513, 8), (1, 16, 385, 64)])
def test_edges(scheme, B, H, n, d):
    _close(*_run(B, H, n, d, scheme))


@pytest.mark.parametrize("scheme", [oracle.FULL, oracle.MASKED])
def test_rising_keys(scheme):
    # every block raises the running maxima (a factor per key: scores of up to about 60)
    n = 640

    def grow(t):
        t[1] *= (1.0 + 2.0 * np.arange(n, dtype=np.float32) / 128)[None, :, None, None]
    got, ref = _run(1, 12, n, 64, scheme, grow)
    _close(got, ref, 2e-5)           # (scores of 60: 2^-24 * 61 = 3.6e-6 per weight, five times over)


@pytest.mark.parametrize("scheme", [oracle.FULL, oracle.MASKED])
def test_heads_with_numbers_without_parts(scheme):
    # head 1: one infinite key, head 2: values around 1e-30, head 3: one value of 1e25; heads 0 and 4 must not notice
    B, H, n, d = 3, 5, 600, 64

    def spoil(t):
        t[1][1, 590, 1, 3] = np.inf
        t[2][:, :, 2] *= np.float32(1e-30)
        t[2][0, 7, 3, 5] = np.float32(1e25)
    got, ref = _run(B, H, n, d, scheme, spoil)
    got, ref = got.reshape(B, n, H, d), ref.reshape(B, n, H, d)
    for h in (0, 2, 4):
        _close(got[:, :, h], ref[:, :, h])
    _close(got[0, :, 1], ref[0, :, 1])
    _close(got[:, :, 3][:, :, :5], ref[:, :, 3][:, :, :5])


# Values up to and beyond the largest that the parts carry (2^46), all of one sign, under weights of up to e^3.9 relative to the running maximum, which
# follows only a growth by more than 4: FULL through its first 64 keys, MASKED through the diagonal tile of the last 128 rows.  The
# running sum of 832 such values was infinite from 2^48.6 on.
@pytest.mark.parametrize("scheme", [oracle.FULL, oracle.MASKED])
@pytest.mark.parametrize("power", [45, 46, 47, 49, 50, 60])
def test_large_values_under_a_lagging_maximum(scheme, power):
    B, H, n, d = 1, 16, 1024, 64

    def set_up(t):
        t[0][:], t[1][:] = 0.0, 0.0
        t[0][..., 0] = 8.0                       # 1 / sqrt(d) = 1/8: a key's score is its first number
        t[1][:, 64:n - 128, :, 0] = 3.9
        t[2][:] = np.float32(2.0 ** power) * (1.0 - 0.5 * np.abs(t[2]) / np.abs(t[2]).max())
    got, ref = _run(B, H, n, d, scheme, set_up)
    _close(got / 2.0 ** power, ref / 2.0 ** power)


# The same calls on the tensor cores and, in a registered workspace without room for their operands, on CUDA cores: the error against 64 bits is not
# larger (5 % for the draw).  Values of one sign show sums that are rounded in long chains.
@pytest.mark.parametrize("positive", [False, True])
@pytest.mark.parametrize("H,n,d,scheme", [(40, 257, 64, oracle.MASKED), (31, 300, 128, oracle.MASKED), (8, 768, 128, oracle.MASKED), (16, 1024, 128, oracle.MASKED),
                                          (48, 512, 64, oracle.FULL), (60, 193, 128, oracle.FULL), (2, 1024, 64, oracle.FULL)])
def test_error_is_not_above_that_on_cuda_cores(H, n, d, scheme, positive):
    g = torch.Generator(device="cuda").manual_seed(n + d)
    q, k, v = [torch.empty(1, n, H, d, device="cuda").normal_(generator=g) for _ in range(3)]
    if positive:
        v = v.abs()
    s = torch.einsum("bihc,bjhc->bhij", q.double(), k.double()) / d ** 0.5
    if scheme == oracle.MASKED:
        s = s.masked_fill(~torch.ones(n, n, dtype=torch.bool, device="cuda").tril(), float("-inf"))
    ref = torch.einsum("bhij,bjhc->bihc", torch.softmax(s, -1), v.double()).reshape(1, n, H * d)
    assert binding.psa_workspace_bytes(1, H, n, 0, d, scheme, binding.F32) > 4096          # (a call of the tensor cores)
    error = [float((binding.psa_attention_core(q, k, v, scheme).double() - ref).norm())]
    try:
        binding.psa_set_workspace(torch.empty(4096, dtype=torch.uint8, device="cuda"))
        error.append(float((binding.psa_attention_core(q, k, v, scheme).double() - ref).norm()))
        torch.cuda.synchronize()
    finally:
        binding.psa_set_workspace(None)
    assert error[0] <= 1.05 * error[1], [e / float(ref.norm()) for e in error]


# Projections of the largest calls (pairs of CTAs, 256 x 256 tiles, 64 k at a time): ragged rows, columns and depth, tiny and
# infinite operands.  With one vector per sequence the attention returns V.  Bound: six bf16 products per fp32 product leave 2^-24 of it
# out, sums are rounded every 64 k: (K / 64 + 4) 2^-24 of the sum of magnitudes.
@pytest.mark.parametrize("rows,D,H,d", [(2100, 776, 33, 32), (4111, 328, 16, 64), (2048, 768, 12, 64)])
def test_projections_of_large_calls(rows, D, H, d):
    X, Wq, Wk, Wv = [inputs.tensor(rows + D, i, s, 1.0, "f32")[1] for i, s in enumerate([(rows, 1, D)] + [(D, H * d)] * 3)]
    X[7] *= np.float32(1e-36)
    X[300, 0, 5] = np.inf
    z = binding.psa_attention_f32(*[torch.from_numpy(t).cuda() for t in (X, Wq, Wk, Wv)], H, binding.FULL)
    st, got = binding.psa_last_issued()
    assert st == binding.OK and got == binding.psa_skip_count(rows, H, 1, D, d, binding.FULL, binding.F32)
    z, x, w = z.cpu().numpy().reshape(rows, H * d).astype(np.float64), X.reshape(rows, D).astype(np.float64), Wv.astype(np.float64)
    assert not np.isfinite(z[300]).all()
    x[300], z[300] = 0.0, 0.0
    assert (np.abs(z - x @ w) <= (D / 64 + 4) * 2.0 ** -24 * (np.abs(x) @ np.abs(w)) + 1e-44).all()


@pytest.mark.parametrize("scheme", [oracle.FULL, oracle.MASKED])
@pytest.mark.parametrize("B,H,n,d", [(1, 16, 1024, 64), (2, 10, 700, 128), (1, 4, 300, 64), (1, 3, 70, 20)])
def test_output_over_q(scheme, B, H, n, d):
    # in place, on the tensor cores or not: both results are within 4e-6 of the exact one
    t = [torch.from_numpy(inputs.tensor(n + d, 4 + i, (B, n, H, d), 1.0, "f32")[1]).cuda() for i in range(3)]
    want = binding.psa_attention_core(*t, scheme).double()
    got = binding.psa_attention_core(*t, scheme, out=t[0].view(B, n, H * d)).double()
    st, census = binding.psa_last_issued()
    assert st == binding.OK and census == binding.psa_skip_count(B, H, n, 0, d, scheme, binding.F32)
    assert float((got - want).norm()) <= 8e-6 * float(want.norm())


def test_projections_of_host_calls_in_parts():
    # 8 parts of 2048 rows, on pairs of CTAs each; numbers without parts in the first and the last; bit by bit what the device call gives
    rows, D, H, d = 16384, 768, 12, 64
    X, Wq, Wk, Wv = [torch.from_numpy(inputs.tensor(3, i, s, 1.0, "f32")[1]).pin_memory() for i, s in enumerate([(rows, 1, D)] + [(D, H * d)] * 3)]
    X[7] *= 1e-36
    X[rows - 1, 0, :5] = 1e-33
    out = torch.empty((rows, 1, H * d)).pin_memory()
    binding.psa_attention_host(X, Wq, Wk, Wv, H, binding.FULL, out)
    st, got = binding.psa_last_issued()
    assert st == binding.OK and got == binding.psa_skip_count(rows, H, 1, D, d, binding.FULL, binding.F32)
    want = binding.psa_attention_f32(X.cuda(), Wq.cuda(), Wk.cuda(), Wv.cuda(), H, binding.FULL)
    assert torch.equal(out, want.cpu())


@pytest.mark.parametrize("rows,D,H,d", [(2056, 768, 12, 64), (2100, 328, 16, 64), (1030, 776, 33, 32)])
def test_all_three_projections_of_large_calls(rows, D, H, d):
    # two vectors per sequence: the weights depend on q and k, so that a wrong tile of any of the three shows.  Scores of size 1 to 5:
    # 2^-24 times that and the projections' error, 4e-6 as above
    X, Wq, Wk, Wv = [inputs.tensor(rows + D, i, s, f, "f32")[1] for i, (s, f) in enumerate([((rows, 2, D), 1.0)] + [((D, H * d), D ** -0.5)] * 3)]
    X[7] *= np.float32(1e-36)
    Wq[3, :40] *= np.float32(1e-36)
    Wk[5, -40:] *= np.float32(1e-36)
    z = binding.psa_attention_f32(*[torch.from_numpy(t).cuda() for t in (X, Wq, Wk, Wv)], H, binding.FULL)
    st, got = binding.psa_last_issued()
    assert st == binding.OK and got == binding.psa_skip_count(rows, H, 2, D, d, binding.FULL, binding.F32)
    q, k, v = [(X.astype(np.float64).reshape(2 * rows, D) @ W.astype(np.float64)).reshape(rows, 2, H, d) for W in (Wq, Wk, Wv)]
    s = np.einsum("bihc,bjhc->bhij", q, k) / np.sqrt(d)
    w = np.exp(s - s.max(-1, keepdims=True))
    ref = np.einsum("bhij,bjhc->bihc", w / w.sum(-1, keepdims=True), v).reshape(rows, 2, H * d)
    _close(z.cpu().numpy().astype(np.float64), ref)


@pytest.mark.parametrize("residual", [False, True])
@pytest.mark.parametrize("rows,D,H,d", [(4111, 768, 12, 64), (6500, 328, 9, 40)])
def test_output_projection_of_large_blocks(rows, D, H, d, residual):
    # one vector per sequence: y = X Wv.  Bound: that of the projections twice, the first one carried through |Wo|, and the rounding of z
    X, Wq, Wk, Wv, Wo = [inputs.tensor(rows + D, i, s, f, "f32")[1] for i, (s, f) in
                         enumerate([((rows, 1, D), 1.0)] + [((D, H * d), D ** -0.5)] * 3 + [((H * d, D), (H * d) ** -0.5)])]
    X[7] *= np.float32(1e-36)
    X[300, 0, 5] = np.inf
    Wo[9, 20:60] *= np.float32(1e-36)
    R = inputs.tensor(rows, 9, (rows, 1, D), 1.0, "f32")[1]
    dev = [torch.from_numpy(t).cuda() for t in (X, Wq, Wk, Wv, Wo, R)]
    z = binding.psa_attention_block(*dev[:5], H, binding.FULL, residual=dev[5] if residual else None)
    st, _ = binding.psa_last_issued()
    assert st == binding.OK
    z = z.cpu().numpy().reshape(rows, D).astype(np.float64)
    assert not np.isfinite(z[300]).any()
    x, wv, wo, r = X.reshape(rows, D).astype(np.float64), Wv.astype(np.float64), Wo.astype(np.float64), R.reshape(rows, D).astype(np.float64) * residual
    x[300], z[300], r[300] = 0.0, 0.0, 0.0
    y = x @ wv
    ey = (D / 64 + 4) * 2.0 ** -24 * (np.abs(x) @ np.abs(wv))
    ref = y @ wo + r
    bound = ey @ np.abs(wo) + (H * d / 64 + 4) * 2.0 ** -24 * ((np.abs(y) + ey) @ np.abs(wo)) + 2.0 ** -23 * np.abs(ref) + 1e-44
    assert (np.abs(z - ref) <= bound).all()
