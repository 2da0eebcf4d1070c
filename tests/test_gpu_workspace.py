"""fp32 calls in a registered workspace that holds everything but the operands of the tensor cores: nothing is allocated, the call runs on CUDA
cores, and a captured graph stays in that workspace.  Reference: the same call in a workspace of psa_workspace_bytes, on the tensor cores; both
are within 4e-6 of the exact result (tests/test_gpu_f32_tensor.py), so 8e-6 apart at most."""
import pytest
import torch

from paper_2012_01114_b200 import binding

pytestmark = pytest.mark.gpu
COUNTERS = 256


def _up(v):
    return (v + 255) // 256 * 256


def _inputs(shapes):
    g = torch.Generator(device="cuda").manual_seed(5)
    return [torch.empty(s, device="cuda").normal_(0.0, scale, generator=g) for s, scale in shapes]


def _close(a, b):
    assert torch.isfinite(a).all()
    assert float((a.double() - b.double()).norm()) <= 8e-6 * float(b.double().norm())


def _case(entry, scheme):
    """The call, the bytes of its lean layout, the census it must show."""
    if entry == "core":
        B, H, n, d = 2, 20, 520, 64
        t = _inputs([((B, n, H, d), 1.0)] * 3)
        return lambda out: binding.psa_attention_core(*t, scheme, out=out), (B, n, H * d), COUNTERS, (B, H, n, 0, d)
    B, H, n, d, D = 4, 12, 520, 64, 768
    t = _inputs([((B, n, D), 1.0)] + [((D, H * d), D ** -0.5)] * 3 + [((H * d, D), (H * d) ** -0.5)])
    lean = COUNTERS + 3 * _up(4 * B * n * H * d)
    if entry == "layer":
        return lambda out: binding.psa_attention_f32(*t[:4], H, scheme, out=out), (B, n, H * d), lean, (B, H, n, D, d)
    return (lambda out: binding.psa_attention_block(*t, H, scheme, out=out, residual=t[0]), (B, n, D), lean + _up(4 * B * n * H * d), (B, H, n, D, d))


@pytest.mark.parametrize("scheme", [binding.FULL, binding.MASKED])
@pytest.mark.parametrize("entry", ["core", "layer", "block"])
def test_small_registered_workspace(entry, scheme):
    call, shape, lean, (B, H, n, D, d) = _case(entry, scheme)
    whole = binding.psa_workspace_bytes(B, H, n, D, d, scheme, binding.F32) if entry != "block" else binding.psa_block_workspace_bytes(B, H, n, D, d, scheme, binding.F32)
    assert lean < whole
    outs = [torch.full(shape, float("nan"), device="cuda") for _ in range(3)]
    big = torch.empty(whole, dtype=torch.uint8, device="cuda")
    small = torch.full((lean + 4096,), 171, dtype=torch.uint8, device="cuda")
    try:
        binding.psa_set_workspace(big)
        call(outs[0])
        binding.psa_set_workspace(small[:lean])
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        call(outs[1])
        st, got = binding.psa_last_issued()
        # (a kernel's first launch may take a little memory; the whole layouts are 16 MB and more)
        assert st == binding.OK and free - torch.cuda.mem_get_info()[0] < 8 << 20 and whole > 15 << 20
        assert not (small[:COUNTERS] == 171).all() and (small[lean:] == 171).all()        # this memory was used, and nothing behind it
        want = binding.psa_skip_count(B, H, n, D, d, scheme, binding.F32)
        assert {k: v for k, v in got.items() if k != "proj_macs"} == {k: v for k, v in want.items() if k != "proj_macs"}
        _close(outs[1], outs[0])
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            call(outs[2])
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(outs[2], outs[1])
    finally:
        torch.cuda.synchronize()
        binding.psa_set_workspace(None)


def test_too_small_even_for_the_lean_layout():
    call, shape, lean, _ = _case("layer", binding.FULL)
    small = torch.empty(lean - 256, dtype=torch.uint8, device="cuda")
    a, b = torch.empty(shape, device="cuda"), torch.empty(shape, device="cuda")
    call(a)
    try:
        binding.psa_set_workspace(small)
        call(b)                                              # in the library's own, on the tensor cores
        torch.cuda.synchronize()
    finally:
        binding.psa_set_workspace(None)
    assert torch.equal(a, b)


@pytest.mark.parametrize("entry", ["core", "layer"])
def test_nothing_is_left_from_call_to_call(entry):
    # Nothing is cleared ahead of a call: heads marked by one call (values of 1e20, weights of 1e-30) are not marked in the next, memory full of anything is no
    # mark, and the census of each call is its own.  The same kernels run on the same numbers, so outputs are equal bit by bit.
    scheme = binding.MASKED if entry == "core" else binding.FULL
    call, shape, _, (B, H, n, D, d) = _case(entry, scheme)
    want = torch.empty(shape, device="cuda")
    call(want)
    bytes_ = binding.psa_workspace_bytes(B, H, n, D, d, scheme, binding.F32)
    if entry == "core":
        q, k, v = _inputs([((B, n, H, d), 1.0)] * 3)
        v[0, 3, 2] = 1e20
        odd = lambda: binding.psa_attention_core(q, k, v, scheme)
    else:
        t = _inputs([((B, n, D), 1.0)] + [((D, H * d), D ** -0.5)] * 3)
        t[1][5, ::3] = 1e-30
        odd = lambda: binding.psa_attention_f32(*t, H, scheme)
    small = _inputs([((3, 40, 4, 32), 1.0)] * 3)
    try:
        for fill in (0x5a, 0x00, 0xff):
            binding.psa_set_workspace(torch.full((bytes_,), fill, dtype=torch.uint8, device="cuda"))
            for before in (lambda: None, odd, odd, lambda: binding.psa_attention_core(*small, binding.FULL), lambda: binding.psa_attention_core(small[0], None, None, binding.SYMMETRIC)):
                before()
                out = torch.full(shape, float("nan"), device="cuda")
                call(out)
                st, got = binding.psa_last_issued()
                assert st == binding.OK and got == binding.psa_skip_count(B, H, n, D, d, scheme, binding.F32)
                assert torch.equal(out.view(torch.int32), want.view(torch.int32))
    finally:
        binding.psa_set_workspace(None)


# What a program may do with a registered workspace between calls: write anywhere but into the first 256 bytes, and there too if it registers the memory again.
@pytest.mark.parametrize("dtype,scheme,entry,B,H,n,D,d", [
    (binding.F32, binding.MASKED, "core", 2, 20, 520, 0, 64), (binding.F32, binding.FULL, "layer", 4, 12, 520, 768, 64), (binding.F32, binding.MASKED, "layer", 1, 1, 64, 64, 64),
    (binding.F32, binding.SYMMETRIC, "core", 2, 3, 100, 0, 32), (binding.F32, binding.FULL, "core", 2, 3, 30, 0, 20), (binding.F32, binding.FULL, "block", 4, 12, 520, 768, 64),
    (binding.BF16, binding.MASKED, "core", 10, 16, 300, 0, 64), (binding.BF16, binding.FULL, "layer", 3, 2, 200, 128, 192), (binding.BF16, binding.SYMMETRIC, "core", 20, 16, 300, 0, 128)])
def test_memory_used_for_other_things_between_calls(dtype, scheme, entry, B, H, n, D, d):
    sym, dt = scheme == binding.SYMMETRIC, torch.bfloat16 if dtype == binding.BF16 else torch.float32
    if entry == "core":
        t = [x.to(dt) for x in _inputs([((B, n, H, d), 1.0)] * (1 if sym else 3))]
        call = lambda: binding.psa_attention_core(*(t + [None, None] if sym else t), scheme)
    else:
        t = [x.to(dt) for x in _inputs([((B, n, D), 1.0)] + [((D, H * d), D ** -0.5)] * 3 + [((H * d, D), (H * d) ** -0.5)])]
        layer = binding.psa_attention if dtype == binding.BF16 else binding.psa_attention_f32
        call = (lambda: binding.psa_attention_block(*t, H, scheme)) if entry == "block" else (lambda: layer(*t[:4], H, scheme))
    size = binding.psa_block_workspace_bytes if entry == "block" else binding.psa_workspace_bytes
    ws = torch.zeros(size(B, H, n, D, d, scheme, dtype), dtype=torch.uint8, device="cuda")

    def checked():
        out = call()
        st, got = binding.psa_last_issued()
        census = binding.psa_skip_count(B, H, n, D, d, scheme, dtype)
        if entry == "block":
            census["proj_macs"] += B * n * H * d * D
        assert st == binding.OK and got == census
        return out.view(torch.int16)
    try:
        binding.psa_set_workspace(ws)
        want = checked()
        for fill in (0xff, 0x5a, 0x00, 0xff):
            ws[COUNTERS:] = fill
            assert torch.equal(checked(), want)
            ws[:] = fill
            binding.psa_set_workspace(ws)
            assert torch.equal(checked(), want)
    finally:
        binding.psa_set_workspace(None)


# Marks of an output projection: those of one call (entries of 1e-30 in Wo) are none in the next, nor in a replay of a graph that has run with
# such entries; the layer in several launches and, 400 sequences of 64 vectors, in one.
@pytest.mark.parametrize("B,H,n,D,d", [(4, 12, 520, 768, 64), (400, 16, 64, 256, 16)])
def test_marks_of_an_output_projection_from_call_to_call(B, H, n, D, d):
    t = _inputs([((B, n, D), 1.0)] + [((D, H * d), D ** -0.5)] * 3 + [((H * d, D), (H * d) ** -0.5)])
    Wo, out = t[4], torch.empty((B, n, D), device="cuda")
    odd = Wo.clone()
    odd[5, ::3] = 1e-30
    call = lambda wo: binding.psa_attention_block(*t[:4], wo, H, binding.FULL, out=out, residual=t[0])
    call(odd)
    marked = out.clone()
    for _ in range(3):
        call(Wo)
    want = out.clone()
    bytes_ = binding.psa_block_workspace_bytes(B, H, n, D, d, binding.FULL, binding.F32)
    try:
        for fill in (0x5a, 0x00, 0xff):
            binding.psa_set_workspace(torch.full((bytes_,), fill, dtype=torch.uint8, device="cuda"))
            for before in ((), (odd,), (odd, odd)):
                for w in before:
                    call(w)
                    assert torch.equal(out, marked)
                call(Wo)
                assert torch.equal(out, want)
        moving = Wo.clone()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            call(moving)
        for wo, expected in ((Wo, want), (odd, marked), (Wo, want), (odd, marked), (Wo, want)):
            moving.copy_(wo)
            out.fill_(float("nan"))
            graph.replay()
            assert torch.equal(out, expected)
            call(wo)
            assert torch.equal(out, expected)
    finally:
        torch.cuda.synchronize()
        binding.psa_set_workspace(None)
