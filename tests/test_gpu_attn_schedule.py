"""Attention with whole query tiles dealt to the persistent blocks before the
rest is cut (more than a wave and a half of tiles), and the merges of shared
tiles, against the fp64 oracle's rows: several waves with ragged last tiles and
empty tails, lengths so uneven that nothing is dealt, decode steps whose tiles
hold a single token and are split over many blocks."""
import numpy as np
import pytest

from workload import synth as W

pytestmark = pytest.mark.gpu
TOL = 5e-3          # the library's bar: bf16 inputs and probabilities, fp32 sums


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_18935_gb300 import kvm
    kvm.load_library()


CASES = {
    # 40 characters x 4 KV heads x up to 8 tiles of 16 tokens: several waves
    "waves": (32, 4, 64, [150 + 7 * b for b in range(40)], [0 if b == 3 else 128 - b for b in range(40)]),
    "waves_d256": (16, 2, 256, [64 + 11 * b for b in range(24)], [97 + b for b in range(24)]),
    "uneven": (32, 4, 64, [12000] + [5] * 39, [128] * 40),
    "short": (16, 2, 256, [0, 70, 300], [16, 1, 20]),          # at most five key tiles: a block a tile
    "decode_one": (16, 2, 256, [6000], [1]),
    "decode_many": (16, 4, 128, [900 + 131 * b for b in range(9)], [1, 2, 0, 1, 1, 3, 1, 1, 1]),
}


@pytest.mark.parametrize("name", CASES)
def test_scheduled_attention_matches_the_oracle(name):
    import torch
    from harness import rel_l2, to_torch_bf16, torch_bf16_to_f64
    from oracle import kvm_oracle as O
    from paper_2609_18935_gb300 import kvm
    hq, hkv, d, live, tails = CASES[name]
    B, n = len(live), sum(tails)
    cu = np.concatenate([[0], np.cumsum(tails)]).astype(np.int32)
    ctx = kvm.Context([kvm.LAYER_ATTN], hq, hkv, d, 64, 1e4, 8, 64, 64, [l + 128 for l in live], n)
    cache = []
    for b, l in enumerate(live):
        ctx.load_prefix(b, l, l, np.arange(l, dtype=np.int32))
        K = W.normal_bf16((81, b, 0), (hkv, l, d), unit_last=True)
        V = W.normal_bf16((81, b, 1), (hkv, l, d))
        ctx.set_kv(0, b, to_torch_bf16(K).cuda(), to_torch_bf16(V).cuda())
        cache.append((K, V))
    q = W.normal_bf16((82, 0), (n, hq, d))
    k = W.normal_bf16((82, 1), (n, hkv, d), unit_last=True)
    v = W.normal_bf16((82, 2), (n, hkv, d))
    dev = [to_torch_bf16(x).cuda() for x in (q, k, v)]
    torch.cuda.synchronize()
    outs = []
    for _ in range(2):                              # the partials' workspace is reused
        out = torch.full((n, hq, d), float("nan"), dtype=torch.bfloat16, device="cuda")
        ctx.tail_attn_prefill(0, cu, *dev, out)
        outs.append(out)
    ctx.check()
    assert torch.equal(outs[0].view(torch.int16), outs[1].view(torch.int16))
    got = torch_bf16_to_f64(outs[0])
    assert np.isfinite(got).all()
    for b in range(B):
        s = slice(cu[b], cu[b + 1])
        if not tails[b]:
            continue
        pos = live[b] + np.arange(tails[b])
        qr = O.rope(O.bf16_to_f64(q[s]), pos, 64, 1e4)
        kr = O.rope(O.bf16_to_f64(k[s]), pos, 64, 1e4)
        K = np.concatenate([O.bf16_to_f64(cache[b][0]), kr.transpose(1, 0, 2)], 1)
        V = np.concatenate([O.bf16_to_f64(cache[b][1]), O.bf16_to_f64(v[s]).transpose(1, 0, 2)], 1)
        want = np.empty_like(got[s])
        for h in range(hq):
            w = qr[:, h] @ K[h // (hq // hkv)].T / np.sqrt(d)
            w[np.arange(K.shape[1])[None, :] > pos[:, None]] = -np.inf
            w = np.exp(w - w.max(1, keepdims=True))
            want[:, h] = (w / w.sum(1, keepdims=True)) @ V[h // (hq // hkv)]
        assert rel_l2(got[s], want) <= TOL, b
