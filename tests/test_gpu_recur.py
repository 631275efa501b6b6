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
