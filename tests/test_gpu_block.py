"""Attention block (layer + output projection over the concatenated heads) against the oracle, both
storage types: values within the paths' tolerances, projection MACs bit-exact."""
import numpy as np
import pytest
import torch

import oracle
from paper_2012_01114_b200 import binding, inputs

pytestmark = pytest.mark.gpu
# bf16 storage, fp32 accumulation: the layer's tolerance (2e-2 on y, which the output projection with a matrix of
# N(0,1)/sqrt(heads*d_k) entries carries over at the same size) plus the rounding of z itself to bf16, at most
# 2^-8 |z| (z reaches 4 and more in the symmetric scheme, where half a bf16 step is already 1.6e-2).
TOL_BF16 = 2e-2
TOL_BF16_REL = 2.0 ** -8
TOL_F32 = 1e-4    # fp32 storage and arithmetic


def _dev_bf16(bits):
    return torch.from_numpy(np.ascontiguousarray(bits).view(np.int16)).cuda().view(torch.bfloat16)


def _to_f64(t):
    return t.float().cpu().numpy().astype(np.float64)


def _proj_macs(B, H, n, D, d, scheme):
    return ((1 if scheme == oracle.SYMMETRIC else 3) + 1) * B * n * D * H * d


@pytest.mark.parametrize("scheme", [oracle.FULL, oracle.MASKED])
def test_block_bf16_with_wide_heads(scheme):
    # heads of 256 columns run on the one-row-tile kernel between the two projection launches
    test_block_bf16_matches_oracle(scheme, 2, 2, 300, 128, 256)
    test_block_bf16_matches_oracle(scheme, 1, 1, 257, 64, 192)


@pytest.mark.parametrize("scheme", [oracle.FULL, oracle.MASKED, oracle.SYMMETRIC])
@pytest.mark.parametrize("B,H,n,D,d", [(1, 1, 128, 64, 64), (2, 3, 256, 192, 64), (1, 2, 384, 320, 128),
                                       (2, 2, 333, 128, 64), (1, 12, 512, 768, 64)])
def test_block_bf16_matches_oracle(scheme, B, H, n, D, d):
    sym = scheme == oracle.SYMMETRIC
    Xv, Xb = inputs.tensor(11, 0, (B, n, D), 1.0, "bf16")
    W = [inputs.tensor(11, 1 + i, (D, H * d), D ** -0.5, "bf16") for i in range(3)]
    Wov, Wob = inputs.tensor(11, 8, (H * d, D), (H * d) ** -0.5, "bf16")
    out = binding.psa_attention_block(_dev_bf16(Xb), _dev_bf16(W[0][1]), None if sym else _dev_bf16(W[1][1]),
                                      None if sym else _dev_bf16(W[2][1]), _dev_bf16(Wob), H, scheme)
    assert tuple(out.shape) == (B, n, D)
    ref, _, _ = oracle.attention_block(Xv, W[0][0], W[1][0], W[2][0], Wov, H, scheme)
    excess = (np.abs(_to_f64(out) - ref) - TOL_BF16_REL * np.abs(ref)).max()
    assert excess <= TOL_BF16, excess
    st, got = binding.psa_last_issued()
    assert st == binding.OK
    assert got["proj_macs"] == _proj_macs(B, H, n, D, d, scheme)
    layer = binding.psa_skip_count(B, H, n, D, d, scheme, binding.BF16)
    for k in ("qk_macs", "pv_macs", "useful_qk_macs", "useful_pv_macs"):
        assert got[k] == layer[k]


@pytest.mark.parametrize("scheme", [oracle.FULL, oracle.MASKED, oracle.SYMMETRIC])
@pytest.mark.parametrize("B,H,n,D,d", [(1, 1, 1, 8, 4), (2, 3, 37, 50, 20), (1, 2, 200, 64, 128)])
def test_block_f32_matches_oracle(scheme, B, H, n, D, d):
    rng = np.random.default_rng(3 * n + d)
    X = (rng.standard_normal((B, n, D)) * 0.5).astype(np.float32)
    Ws = [(rng.standard_normal((D, H * d)) / np.sqrt(D)).astype(np.float32) for _ in range(3)]
    Wo = (rng.standard_normal((H * d, D)) / np.sqrt(H * d)).astype(np.float32)
    sym = scheme == oracle.SYMMETRIC
    dev = lambda a: torch.from_numpy(a).cuda()
    out = binding.psa_attention_block(dev(X), dev(Ws[0]), None if sym else dev(Ws[1]), None if sym else dev(Ws[2]),
                                      dev(Wo), H, scheme)
    ref, _, cnt = oracle.attention_block(X, Ws[0], Ws[1], Ws[2], Wo, H, scheme)
    err = np.abs(out.cpu().numpy().astype(np.float64) - ref).max()
    assert err <= TOL_F32, err
    st, got = binding.psa_last_issued()
    assert st == binding.OK
    assert got["proj_macs"] == _proj_macs(B, H, n, D, d, scheme)
    assert (got["qk_macs"], got["pv_macs"]) == (cnt.mac1, cnt.mac3)


def test_block_equals_layer_then_identity_and_leaves_the_layer_path_alone():
    # Wo = identity (exact in bf16): the block's output is the layer's output bit for bit; calls of the two entry
    # points in turn share the workspace and the counter blocks.
    B, H, n, D, d = 2, 2, 384, 128, 64
    _, Xb = inputs.tensor(12, 0, (B, n, D), 1.0, "bf16")
    W = [_dev_bf16(inputs.tensor(12, 1 + i, (D, H * d), D ** -0.5, "bf16")[1]) for i in range(3)]
    X = _dev_bf16(Xb)
    eye = torch.eye(H * d, dtype=torch.bfloat16, device="cuda")
    for scheme in (oracle.MASKED, oracle.FULL, oracle.MASKED):
        y = binding.psa_attention(X, W[0], W[1], W[2], H, scheme)
        st, c_layer = binding.psa_last_issued()
        z = binding.psa_attention_block(X, W[0], W[1], W[2], eye, H, scheme)
        st2, c_block = binding.psa_last_issued()
        assert st == binding.OK and st2 == binding.OK
        assert torch.equal(y, z)
        assert c_block["proj_macs"] == c_layer["proj_macs"] + B * n * H * d * D
        assert c_block["qk_macs"] == c_layer["qk_macs"] and c_block["pv_macs"] == c_layer["pv_macs"]


def test_block_workspace_and_argument_errors():
    B, H, n, D, d = 1, 2, 256, 128, 64
    need = binding.psa_block_workspace_bytes(B, H, n, D, d, oracle.FULL, binding.BF16)
    assert need >= binding.psa_workspace_bytes(B, H, n, D, d, oracle.FULL, binding.BF16) + B * n * H * d * 2
    L = binding.lib()
    x = torch.zeros((B, n, D), dtype=torch.bfloat16, device="cuda")
    w = torch.zeros((D, H * d), dtype=torch.bfloat16, device="cuda")
    p = lambda t: t.data_ptr()
    args = (B, H, n, D, d, int(oracle.FULL), binding.BF16, p(x), None)
    assert L.psa_attention_block(p(x), p(w), p(w), p(w), None, *args) == binding.ERR_NULL          # no Wo
    assert L.psa_attention_block(p(x), p(w), p(w), p(w), p(w) + 2, *args) == binding.ERR_ALIGN
    bad = (B, H, n, D, 48, int(oracle.FULL), binding.BF16, p(x), None)
    assert L.psa_attention_block(p(x), p(w), p(w), p(w), p(w), *bad) == binding.ERR_UNSUPPORTED
    sym = (B, H, n, D, d, int(oracle.SYMMETRIC), binding.BF16, p(x), None)
    w2 = torch.zeros_like(w)
    assert L.psa_attention_block(p(x), p(w), p(w2), None, p(w), *sym) == binding.ERR_SCHEME_ARGS


@pytest.mark.parametrize("scheme", [oracle.FULL, oracle.MASKED, oracle.SYMMETRIC])
@pytest.mark.parametrize("B,H,n,D,d", [(1, 1, 128, 64, 64), (2, 3, 256, 192, 64), (2, 2, 333, 128, 64), (1, 2, 384, 320, 128)])
def test_block_with_residual_bf16_matches_oracle(scheme, B, H, n, D, d):
    # z = R + y Wo with R = X (the usual skip connection) and with an unrelated R; the sum is formed in fp32 before
    # the rounding of z, so the tolerance is that of the block
    sym = scheme == oracle.SYMMETRIC
    Xv, Xb = inputs.tensor(21, 0, (B, n, D), 1.0, "bf16")
    W = [inputs.tensor(21, 1 + i, (D, H * d), D ** -0.5, "bf16") for i in range(3)]
    Wov, Wob = inputs.tensor(21, 8, (H * d, D), (H * d) ** -0.5, "bf16")
    Rv, Rb = inputs.tensor(21, 9, (B, n, D), 2.0, "bf16")
    X = _dev_bf16(Xb)
    for res_v, res_dev in ((Xv, X), (Rv, _dev_bf16(Rb))):
        out = binding.psa_attention_block(X, _dev_bf16(W[0][1]), None if sym else _dev_bf16(W[1][1]),
                                          None if sym else _dev_bf16(W[2][1]), _dev_bf16(Wob), H, scheme, residual=res_dev)
        ref, _, _ = oracle.attention_block(Xv, W[0][0], W[1][0], W[2][0], Wov, H, scheme, residual=res_v)
        excess = (np.abs(_to_f64(out) - ref) - TOL_BF16_REL * np.abs(ref)).max()
        assert excess <= TOL_BF16, excess
        st, got = binding.psa_last_issued()
        assert st == binding.OK and got["proj_macs"] == _proj_macs(B, H, n, D, d, scheme)


@pytest.mark.parametrize("scheme", [oracle.FULL, oracle.MASKED, oracle.SYMMETRIC])
def test_block_with_residual_f32_matches_oracle(scheme):
    B, H, n, D, d = 2, 3, 37, 50, 20
    rng = np.random.default_rng(77)
    X = (rng.standard_normal((B, n, D)) * 0.5).astype(np.float32)
    Ws = [(rng.standard_normal((D, H * d)) / np.sqrt(D)).astype(np.float32) for _ in range(3)]
    Wo = (rng.standard_normal((H * d, D)) / np.sqrt(H * d)).astype(np.float32)
    R = rng.standard_normal((B, n, D)).astype(np.float32)
    sym = scheme == oracle.SYMMETRIC
    dev = lambda a: torch.from_numpy(a).cuda()
    out = binding.psa_attention_block(dev(X), dev(Ws[0]), None if sym else dev(Ws[1]), None if sym else dev(Ws[2]),
                                      dev(Wo), H, scheme, residual=dev(R))
    ref, _, _ = oracle.attention_block(X, Ws[0], Ws[1], Ws[2], Wo, H, scheme, residual=R)
    assert np.abs(out.cpu().numpy().astype(np.float64) - ref).max() <= TOL_F32


def test_block_residual_must_not_be_the_output():
    B, H, n, D, d = 1, 2, 128, 128, 64
    x = torch.zeros((B, n, D), dtype=torch.bfloat16, device="cuda")
    w = torch.zeros((D, H * d), dtype=torch.bfloat16, device="cuda")
    wo = torch.zeros((H * d, D), dtype=torch.bfloat16, device="cuda")
    out = torch.zeros_like(x)
    with pytest.raises(binding.PsaError) as ei:
        binding.psa_attention_block(x, w, w, w, wo, H, oracle.FULL, out=out, residual=out)
    assert ei.value.status == binding.ERR_SCHEME_ARGS


# The projection kernel has three tiles (128 x 128, 128 x 256, and 256 x 256 over a pair of CTAs), chosen by how many of
# them the call has.  Sequences of one vector make the layer the projection itself (y = v) and the block y Wo + residual:
# rows around the tile edges and the switches, ragged column tiles, one and many k-steps.
@pytest.mark.parametrize("rows,D,H,d", [(1, 64, 1, 64), (129, 128, 2, 64), (257, 192, 5, 64), (1000, 320, 3, 128), (2000, 768, 12, 64),
                                        (4096, 64, 12, 64), (5000, 1024, 7, 64), (9000, 1600, 13, 64), (300, 64, 20, 128)])
def test_projection_tile_choices(rows, D, H, d):
    g = torch.Generator(device="cuda").manual_seed(rows + D)
    X = torch.randn(rows, 1, D, device="cuda", generator=g).bfloat16()
    W = [(torch.randn(D, H * d, device="cuda", generator=g) * D ** -0.5).bfloat16() for _ in range(3)]
    Wo = (torch.randn(H * d, D, device="cuda", generator=g) * (H * d) ** -0.5).bfloat16()
    y = binding.psa_attention(X, *W, H, binding.FULL)
    st, got = binding.psa_last_issued()
    assert st == binding.OK and got["proj_macs"] == 3 * rows * D * H * d
    ref = X.double().view(rows, D) @ W[2].double()
    # one rounding to bf16 of a sum of K products in fp32 (|q|, |k| = O(1): the single weight is exactly 1)
    assert ((y.double().view(rows, -1) - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-4).all()
    z = binding.psa_attention_block(X, *W, Wo, H, binding.FULL, residual=X)
    st, got = binding.psa_last_issued()
    assert st == binding.OK and got["proj_macs"] == 4 * rows * D * H * d
    zref = y.double().view(rows, -1) @ Wo.double() + X.double().view(rows, D)
    assert ((z.double().view(rows, -1) - zref).abs() <= 2.0 ** -8 * zref.abs() + 1e-4).all()


def _near(got, a, w, plus=0.0):
    # a w + plus as summed in fp32 (K 2^-24 of the sum of sizes) and rounded to bf16 (2^-9)
    a, w = a.double(), w.double()
    ref = a @ w + plus
    bound = 2.0 ** -8 * ref.abs() + a.shape[1] * 2.0 ** -24 * (a.abs() @ w.abs())
    assert ((got.double() - ref).abs() <= bound).all()


# One vector per sequence attends to itself: the layer's output is the projection X Wv, the block's that times Wo.  Sizes at which tiles of 192
# columns are chosen, with ragged last tiles of rows and columns.
@pytest.mark.parametrize("M,N,K", [(2048, 512, 512), (1990, 512, 576), (4000, 192, 512), (2700, 320, 512), (1000, 1024, 512), (4090, 768, 768)])
def test_projections_on_tiles_of_192_columns(M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M + N)
    X = torch.randn(M, 1, K, device="cuda", generator=g).bfloat16()
    W = [(torch.randn(K, N, device="cuda", generator=g) * K ** -0.5).bfloat16() for _ in range(3)]
    y = binding.psa_attention(X, *W, N // 64, binding.FULL)
    _near(y[:, 0], X[:, 0], W[2])
    if N == K:
        Wo = (torch.randn(N, K, device="cuda", generator=g) * N ** -0.5).bfloat16()
        for R in (None, X):
            z = binding.psa_attention_block(X, *W, Wo, N // 64, binding.FULL, residual=R)
            _near(z[:, 0], y[:, 0], Wo, 0.0 if R is None else R[:, 0].double())


# The same tiles where the output depends on all three projections, and an output projection with a last tile of columns that is cut short, with and
# without residual: 192 columns at these sizes (tests/test_gemm_tile_cpu.py).  Reference: 64 bits from q, k, v rounded to bf16; bounds as
# elsewhere on this path, 2e-2 and half a bf16 step of the output itself.
@pytest.mark.parametrize("scheme,B,n,K,H", [(binding.FULL, 128, 16, 512, 8), (binding.MASKED, 20, 100, 576, 8), (binding.FULL, 40, 100, 512, 3),
                                            (binding.MASKED, 21, 129, 512, 5), (binding.SYMMETRIC, 80, 100, 512, 11)])
def test_layers_on_tiles_of_192_columns(scheme, B, n, K, H):
    d, N, sym = 64, 64 * H, scheme == binding.SYMMETRIC
    g = torch.Generator(device="cuda").manual_seed(B + n)
    X = torch.randn(B, n, K, device="cuda", generator=g).bfloat16()
    W = [(torch.randn(K, N, device="cuda", generator=g) * K ** -0.5).bfloat16() for _ in range(1 if sym else 3)]
    y = binding.psa_attention(X, *(W + [None, None] if sym else W), H, scheme)
    st, got = binding.psa_last_issued()
    assert st == binding.OK and got == binding.psa_skip_count(B, H, n, K, d, scheme, binding.BF16)
    q, k, v = [(X.double() @ w.double()).bfloat16().double().view(B, n, H, d).transpose(1, 2) for w in (W * 3)[:3]]
    s = q @ k.transpose(2, 3) * d ** -0.5
    if scheme == binding.MASKED:
        s = s.masked_fill(torch.ones(n, n, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    ref = (s.softmax(3) @ v).transpose(1, 2).reshape(B, n, N)
    assert ((y.double() - ref).abs() <= 2e-2 + 2.0 ** -8 * ref.abs()).all()


def test_output_projection_on_tiles_of_192_columns_cut_short():
    M, K, N = 8000, 512, 704
    g = torch.Generator(device="cuda").manual_seed(3)
    X = torch.randn(M, 1, N, device="cuda", generator=g).bfloat16()
    W = [(torch.randn(N, K, device="cuda", generator=g) * N ** -0.5).bfloat16() for _ in range(3)]
    Wo = (torch.randn(K, N, device="cuda", generator=g) * K ** -0.5).bfloat16()
    y = binding.psa_attention(X, *W, K // 64, binding.FULL)
    for R in (None, X):
        z = binding.psa_attention_block(X, *W, Wo, K // 64, binding.FULL, residual=R)
        st, got = binding.psa_last_issued()
        assert st == binding.OK and got["proj_macs"] == 4 * M * K * N
        _near(z[:, 0], y[:, 0], Wo, 0.0 if R is None else R[:, 0].double())
