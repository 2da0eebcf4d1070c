"""Calls captured into CUDA graphs: every replay computes the whole call anew on the inputs of the moment, and neither
replays nor captures disturb the calls made between them (results and census)."""
import pytest
import torch

from paper_2012_01114_b200 import binding

pytestmark = pytest.mark.gpu


def _call(entry, dtype, scheme, B, H, n, d):
    """(input tensors, function of them and an output buffer, output, arguments of the census)"""
    dt = torch.bfloat16 if dtype == binding.BF16 else torch.float32
    g = torch.Generator(device="cuda").manual_seed(n + d)

    def normal(*shape, scale=1.0):
        return (torch.randn(*shape, device="cuda", generator=g) * scale).to(dt)
    sym = scheme == binding.SYMMETRIC
    if entry == "core":
        ins = [normal(B, n, H, d) for _ in range(1 if sym else 3)]
        q = (lambda: (ins[0], None, None)) if sym else (lambda: tuple(ins))
        return ins, lambda out: binding.psa_attention_core(*q(), scheme, out=out), torch.empty(B, n, H * d, dtype=dt, device="cuda"), \
            (B, H, n, 0, d, scheme, dtype)
    D = 128
    W = [normal(D, H * d, scale=D ** -0.5) for _ in range(1 if sym else 3)] + ([None, None] if sym else [])
    Wo = normal(H * d, D, scale=(H * d) ** -0.5)
    ins = [normal(B, n, D)]
    if entry == "block":
        return ins, lambda out: binding.psa_attention_block(ins[0], *W, Wo, H, scheme, out=out), torch.empty(B, n, D, dtype=dt, device="cuda"), None
    layer = binding.psa_attention if dtype == binding.BF16 else binding.psa_attention_f32
    return ins, lambda out: layer(ins[0], *W, H, scheme, out=out), torch.empty(B, n, H * d, dtype=dt, device="cuda"), \
        (B, H, n, D, d, scheme, dtype)


# More work items than SMs, so that the device-side work counter of the fused kernels matters: heads up to 64, 128 and 256
# columns, with and without projections; the symmetric kernel; the fp32 forms.
@pytest.mark.parametrize("entry,dtype,scheme,B,H,n,d", [
    ("core", binding.BF16, binding.MASKED, 8, 8, 1024, 64), ("core", binding.BF16, binding.FULL, 4, 16, 1000, 128),
    ("core", binding.BF16, binding.MASKED, 4, 8, 1024, 256), ("core", binding.BF16, binding.FULL, 30, 8, 200, 192),
    ("core", binding.BF16, binding.SYMMETRIC, 8, 8, 512, 64), ("layer", binding.BF16, binding.MASKED, 20, 4, 512, 128),
    ("block", binding.BF16, binding.FULL, 40, 2, 300, 160), ("layer", binding.F32, binding.MASKED, 1, 1, 64, 64),
    ("layer", binding.F32, binding.FULL, 6, 2, 300, 64), ("core", binding.F32, binding.SYMMETRIC, 2, 4, 200, 32)])
def test_replays(entry, dtype, scheme, B, H, n, d):
    ins, call, out, census = _call(entry, dtype, scheme, B, H, n, d)
    other_ins, other, other_out, other_census = _call("core", binding.BF16, binding.MASKED, 8, 8, 600, 128)

    def eager(f, o):
        return f(o).clone()
    want_other = eager(other, other_out)
    eager(call, out)                          # the workspace has its size, the kernels are set up
    graphs = [torch.cuda.CUDAGraph() for _ in range(2)]
    for gr in graphs:                         # a capture runs nothing; the second call of the pair must not rely on the first
        with torch.cuda.graph(gr):
            call(out)
    eager(other, other_out)
    for step in range(6):
        for t in ins:
            t.copy_(t.roll(step + 1, 1))
        out.fill_(float("nan"))
        graphs[step % 2].replay()
        if step % 3 == 1:
            graphs[0].replay()
        got_out = out.clone()
        assert torch.equal(eager(call, out), got_out), step
        if census:
            st, got = binding.psa_last_issued()
            assert st == binding.OK and got == binding.psa_skip_count(*census)
        for _ in range(step % 3):
            assert torch.equal(eager(other, other_out), want_other)
            st, got = binding.psa_last_issued()
            assert st == binding.OK and got == binding.psa_skip_count(*other_census)


def test_census_of_a_captured_call():
    ins, call, out, census = _call("core", binding.BF16, binding.MASKED, 4, 8, 1024, 256)
    call(out)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(out)
    for _ in range(3):
        graph.replay()
        torch.cuda.synchronize()
        st, got = binding.psa_last_issued()      # the captured call was the last one made
        assert st == binding.OK and got == binding.psa_skip_count(*census)
