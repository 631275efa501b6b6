"""The token-by-token delta rule (short tails) against the fp64 oracle's
recurrence, at the edges of its range: the shortest tails, the staging tile,
the longest tail it takes and the next one (chunked), ragged packs with empty
tails, widths of d_v that admit one, two or four rows a lane group, gates at
their ends."""
import numpy as np
import pytest

from workload import synth as W

pytestmark = pytest.mark.gpu

# bf16 outputs: 8 significant bits, so rounding moves a value by at most 2^-8 of
# it.  State: each of n tokens adds a
# few fp32 roundings of values of the state's size, (n + 8) 2^-24 at most; the
# chunked form's split operands carry ~2^-15 relative per product (5e-6 measured
# at most, 2e-5 allowed).
OUT_TOL = 2.0 ** -8


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_18935_gb300 import kvm
    kvm.load_library()


@pytest.mark.parametrize("gates", ["drawn", "ends"])
@pytest.mark.parametrize("heads,dk,dv", [(16, 128, 128), (8, 64, 64), (3, 64, 96), (2, 128, 32)])
@pytest.mark.parametrize("tails", [[1], [17], [32], [33], [48], [1] * 40, [16, 0, 1, 31, 2] * 5])
def test_short_tails_follow_the_recurrence(heads, dk, dv, tails, gates):
    import torch
    from harness import rel_l2, to_torch_bf16, torch_bf16_to_f64
    from oracle import kvm_oracle as O
    from paper_2609_18935_gb300 import kvm
    n, B = sum(tails), len(tails)
    cu = np.concatenate([[0], np.cumsum(tails)]).astype(np.int32)
    ctx = kvm.Context([kvm.LAYER_GDN], 8, 2, 64, 64, 1e4, heads, dk, dv, [64] * B, n)
    q = W.normal_bf16((71, 0), (n, heads, dk))
    k = W.normal_bf16((71, 1), (n, heads, dk), unit_last=True)
    v = W.normal_bf16((71, 2), (n, heads, dv))
    alpha, beta = W.gates((71, 3), n, heads)
    if gates == "ends":
        alpha[::2], beta[::3] = 1.0, 0.0
    S = W.state_f32((71, 4), (B, heads, dv, dk))
    ctx.set_state(0, torch.from_numpy(S).cuda())
    out = torch.empty((n, heads, dv), dtype=torch.bfloat16, device="cuda")
    dev = [to_torch_bf16(x).cuda() for x in (q, k, v)]
    ctx.gdn_chunk_scan_from_state(0, cu, *dev, torch.from_numpy(alpha).cuda(), torch.from_numpy(beta).cuda(), out)
    ctx.check()
    got_o, got_S = torch_bf16_to_f64(out), ctx.get_state(0).cpu().numpy()
    chunked = max(tails) > (48 if dk == 64 else 32)
    for b in range(B):
        s = slice(cu[b], cu[b + 1])
        o, Sb = O.gdn_recurrent(*(O.bf16_to_f64(x[s]) for x in (q, k, v)), O.f32_to_f64(alpha[s]), O.f32_to_f64(beta[s]),
                                O.f32_to_f64(S[b]))
        if tails[b]:
            assert rel_l2(got_o[s], o) <= OUT_TOL, b
        for h in range(heads):
            assert rel_l2(got_S[b, h], Sb[h]) <= (2e-5 if chunked else (tails[b] + 8) * 2.0 ** -24), (b, h)


def test_an_alpha_of_zero_clears_the_state():
    """The decayed state vanishes exactly: S = beta v k^T after such a token."""
    import torch
    from harness import to_torch_bf16
    from oracle import kvm_oracle as O
    from paper_2609_18935_gb300 import kvm
    H, D = 4, 128
    ctx = kvm.Context([kvm.LAYER_GDN], 8, 2, 64, 64, 1e4, H, D, D, [64], 8)
    ctx.set_state(0, torch.from_numpy(W.state_f32((72, 0), (1, H, D, D))).cuda())
    q, k, v = (W.normal_bf16((72, 1 + i), (1, H, D), unit_last=i == 1) for i in range(3))
    out = torch.empty((1, H, D), dtype=torch.bfloat16, device="cuda")
    beta = np.full((1, H), 0.75, np.float32)
    ctx.gdn_chunk_scan_from_state(0, [0, 1], *(to_torch_bf16(x).cuda() for x in (q, k, v)), torch.zeros(1, H, device="cuda"),
                                  torch.from_numpy(beta).cuda(), out)
    want = 0.75 * O.bf16_to_f64(v)[0][:, :, None] * O.bf16_to_f64(k)[0][:, None, :]
    np.testing.assert_allclose(ctx.get_state(0)[0].cpu().numpy(), want, rtol=2.0 ** -22, atol=0)


@pytest.mark.parametrize("heads,dk,dv", [(4, 64, 96), (3, 128, 128)])
def test_short_tails_after_the_convolution(heads, dk, dv):
    """The convolution inside the step (a few tokens), in a launch before it, and
    before the chunked form, with the carried state passed between them: rounds of
    one population whose tails cross those limits, and empty tails."""
    from harness import Pair
    shape = W.ModelShape([W.GDN, W.GDN], 8, 2, 64, 64, 1e4, heads, dk, dv)
    prefix = [0, 0, 0]
    pair = Pair(shape, prefix, [256] * 3, 160, seed_index=94, conv=True)
    w = W.Workload("recur-conv", 94, shape, prefix, 7)
    for r, tails in enumerate([[1, 2, 0], [4, 3, 1], [0, 0, 2], [5, 9, 32], [33, 1, 0], [1, 1, 1], [48, 49, 2]]):
        w.plan = [[(0.0, 0, m) for m in tails]] * 7
        errs = pair.run_round(np.zeros(4, np.int32), np.zeros(0, np.int32), np.zeros(0, np.int32), tails,
                              W.tail_inputs(w, r, tails))
        bad = {k: v for k, v in errs.items() if not v <= 5e-3}       # the library's bar, bf16 inputs
        assert not bad, (r, bad)


@pytest.mark.parametrize("conv", [False, True])
@pytest.mark.parametrize("tails,over", [(t, o) for t in ([1, 0], [2, 1], [20, 1]) for o in ("v", "q", "k", "v_ahead", "gates")] +
                         [([2048], "q"), ([2048], "q_ahead"), ([2048], "gates")])
def test_outputs_over_the_inputs(tails, over, conv):
    """An out that lies over an input, at its address or four rows before it:
    outputs, state and carried convolution inputs as with an out of its own."""
    import torch
    from paper_2609_18935_gb300 import kvm
    H, D, n, B = 16, 128, sum(tails), len(tails)
    row = H * D
    g = torch.Generator("cuda").manual_seed(8)
    cu = np.concatenate([[0], np.cumsum(tails)])
    x = [torch.randn((n, H, D), generator=g, device="cuda").bfloat16() for _ in range(3)]
    x[1] = (x[1].float() / x[1].float().norm(dim=-1, keepdim=True)).bfloat16()
    gates = torch.sigmoid(torch.randn((2, n, H), generator=g, device="cuda") + 1)
    w = torch.randn((3 * row, 4), generator=g, device="cuda")
    S = 0.2 * torch.randn((B, H, D, D), generator=g, device="cuda")
    got = []
    for shared in (False, True):
        ctx = kvm.Context([kvm.LAYER_GDN], 8, 2, 64, 64, 1e4, H, D, D, [64] * B, n, conv_kernel=4 if conv else 0)
        ctx.set_state(0, S)
        if conv:
            ctx.set_conv_weights(0, w)
        # q, k, v, with room before each, and the gates inside out's bytes
        y = []
        for t in x:
            room = torch.zeros(4 * row + t.numel(), dtype=torch.bfloat16, device="cuda")
            room[4 * row:] = t.flatten()
            y.append(room)
        at = {"q": 0, "k": 1, "v": 2}.get(over[0])
        al, be = gates.clone()
        if over == "gates":
            room = torch.zeros(n * row, dtype=torch.bfloat16, device="cuda")
            al, be = (room[i * n * H * 2:(i + 1) * n * H * 2].view(torch.float32).view(n, H) for i in (0, 1))
            al.copy_(gates[0])
            be.copy_(gates[1])
            out = room
        else:
            out = y[at][:n * row] if over.endswith("ahead") else y[at][4 * row:]
        out = out.view(n, H, D) if shared else torch.empty((n, H, D), dtype=torch.bfloat16, device="cuda")
        torch.cuda.synchronize()
        q, k, v = (t[4 * row:].view(n, H, D) for t in y)
        ctx.gdn_chunk_scan_from_state(0, cu, q, k, v, al, be, out)
        ctx.check()
        got.append((out.float(), ctx.get_state(0), ctx.get_conv_state(0).float() if conv else torch.zeros(1)))
    (o, s, c), (o2, s2, c2) = got
    assert torch.equal(c, c2)
    if (over == "v" and (not conv or max(tails) > 4)) or n > 2000:      # the same kernels, or two forms that agree to the bit
        assert torch.equal(o, o2) and torch.equal(s, s2)
    else:
        # the chunked form for the token-by-token one: an output rounds to bf16 once
        # either way, states differ by the chunked form's 2e-5; a convolution in a
        # launch of its own sums a key's norm in another order, which moves the key by a
        # rounding of bf16, 2^-8
        assert (o - o2).norm() <= 2.0 ** -7 * o.norm()
        assert (s - s2).norm() <= (2.0 ** -8 if conv else 2e-5) * s.norm()


@pytest.mark.parametrize("heads,dk,B,launches", [(16, 128, 1, 3), (16, 128, 16, 1), (16, 64, 1, 1)])
def test_a_decode_step_with_the_state_chain_on(heads, dk, B, launches):
    """The state chain takes a short tail where it can be served (prep, chain and
    outputs); elsewhere the switch changes nothing (one launch, the same bits)."""
    import torch
    from paper_2609_18935_gb300 import kvm
    g = torch.Generator("cuda").manual_seed(9)
    r = lambda *s: torch.randn(s, generator=g, device="cuda")
    q, k, v = r(B, heads, dk).bfloat16(), (r(B, heads, dk) / dk ** 0.5).bfloat16(), r(B, heads, dk).bfloat16()
    al, be, S = torch.sigmoid(r(B, heads)), torch.sigmoid(r(B, heads)), r(B, heads, dk, dk)
    got = []
    for on in (False, True):
        ctx = kvm.Context([kvm.LAYER_GDN], 8, 2, 64, 64, 1e4, heads, dk, dk, [64] * B, B)
        ctx.set_gdn_state_chain(on)
        ctx.set_state(0, S)
        out = torch.empty_like(v)
        before = kvm._lib.kvm_launch_count(ctx._h)
        ctx.gdn_chunk_scan_from_state(0, np.arange(B + 1), q, k, v, al, be, out)
        n = kvm._lib.kvm_launch_count(ctx._h) - before
        ctx.check()
        got.append((out.float(), ctx.get_state(0)))
    assert n == launches
    if n == 1:
        assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    else:
        assert (got[0][1] - got[1][1]).norm() <= 2e-5 * got[0][1].norm()
