"""State accessors: what was set is read back bit for bit, at lengths that are
no multiple of a vector, next to other characters' rows, from buffers on and off
the 16-byte grid, and in order with the calls around them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("live", [[1, 63, 4097], [130, 7, 20001]])
def test_kv_and_positions_round_trip(live, offset):
    import torch
    from paper_2609_18935_gb300 import kvm
    ctx = kvm.Context([kvm.LAYER_GDN, kvm.LAYER_ATTN, kvm.LAYER_ATTN], 8, 2, 64, 64, 1e4, 3, 64, 96, [l + 5 for l in live], 8)
    kept = {}
    for b, l in enumerate(live):
        pos = np.cumsum(np.random.default_rng(b).integers(1, 5, l)).astype(np.int32)
        ctx.load_prefix(b, l, int(pos[-1]) + 1, pos)
        for layer in (1, 2):
            k, v = (torch.randn(2 * l * 64 + offset, device="cuda").bfloat16()[offset:].view(2, l, 64) for _ in range(2))
            ctx.set_kv(layer, b, k, v)
            kept[layer, b] = k, v
        kept["pos", b] = pos
    S = torch.randn(len(live) * 3 * 96 * 64 + offset, device="cuda")[offset:].view(len(live), 3, 96, 64)
    ctx.set_state(0, S)
    assert torch.equal(ctx.get_state(0), S)
    for b, l in enumerate(live):
        assert np.array_equal(ctx.get_positions(b).cpu().numpy(), kept["pos", b])
        for layer in (1, 2):
            for got, want in zip(ctx.get_kv(layer, b), kept[layer, b]):
                assert torch.equal(got.view(torch.int16), want.contiguous().view(torch.int16))


def test_reads_follow_the_writes_queued_before_them():
    """Sets, steps and reads queued without waiting give what they give one by one."""
    import torch
    from paper_2609_18935_gb300 import kvm
    H, D, n = 4, 64, 3
    ctx = kvm.Context([kvm.LAYER_GDN], 8, 2, 64, 64, 1e4, H, D, D, [64], n)
    g = torch.Generator("cuda").manual_seed(1)
    r = lambda *s: torch.randn(s, generator=g, device="cuda")
    q, k, v = r(n, H, D).bfloat16(), r(n, H, D).bfloat16() / 8, r(n, H, D).bfloat16()
    al, be = torch.sigmoid(r(n, H)), torch.sigmoid(r(n, H))
    S = [r(1, H, D, D) for _ in range(8)]
    out = torch.empty_like(v)
    torch.cuda.synchronize()
    runs = []
    for wait in (True, False):
        sync = torch.cuda.synchronize if wait else lambda: None
        got = []
        for s in S:
            ctx.set_state(0, s)
            sync()
            ctx.gdn_chunk_scan_from_state(0, [0, n], q, k, v, al, be, out)
            sync()
            got.append(ctx.get_state(0))
            sync()
        runs.append(got)
    assert all(torch.equal(a, b) for a, b in zip(*runs))


def test_buffers_outside_the_device_are_copied_by_memcpy():
    """Pinned host memory: no kernel of the library reads or writes it
    (the launch count stays), the values arrive all the same."""
    import torch
    from paper_2609_18935_gb300 import kvm
    H, D = 4, 64
    ctx = kvm.Context([kvm.LAYER_GDN, kvm.LAYER_ATTN], 8, 2, 64, 64, 1e4, H, D, D, [128], 8)
    ctx.load_prefix(0, 100, 100, np.arange(100, dtype=np.int32))
    S = torch.randn((1, H, D, D)).pin_memory()
    K, V = (torch.randn((2, 100, 64)).bfloat16().pin_memory() for _ in range(2))
    back = [torch.zeros_like(t).pin_memory() for t in (S, K, V)]
    lib, s = kvm._lib, torch.cuda.current_stream().cuda_stream
    before = lib.kvm_launch_count(ctx._h)
    for call in (lambda: lib.kvm_set_state(ctx._h, 0, S.data_ptr(), s),
                 lambda: lib.kvm_set_kv(ctx._h, 1, 0, K.data_ptr(), V.data_ptr(), s),
                 lambda: lib.kvm_get_state(ctx._h, 0, back[0].data_ptr(), s),
                 lambda: lib.kvm_get_kv(ctx._h, 1, 0, back[1].data_ptr(), back[2].data_ptr(), s)):
        assert call() == 0, lib.kvm_last_error().decode()
    torch.cuda.synchronize()
    assert lib.kvm_launch_count(ctx._h) == before
    for a, b in zip((S, K, V), back):
        assert torch.equal(a, b)
    got = ctx.get_state(0)
    assert lib.kvm_launch_count(ctx._h) == before + 1 and torch.equal(got.cpu(), S)


def test_accessors_under_capture():
    """A captured read replays with the state of the moment."""
    import torch
    from paper_2609_18935_gb300 import kvm
    H, D = 4, 64
    ctx = kvm.Context([kvm.LAYER_GDN], 8, 2, 64, 64, 1e4, H, D, D, [64], 8)
    S = [torch.randn((1, H, D, D), device="cuda") for _ in range(2)]
    ctx.set_state(0, S[0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = ctx.get_state(0)
    for x in S:
        ctx.set_state(0, x)
        graph.replay()
        assert torch.equal(out, x)
