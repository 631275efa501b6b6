"""Two rounds of a stack of one delta-rule layer with nothing between them: the
second round's launch may start before the first has finished, and must still
read the state the first one wrote: as one launch for prep and scan (long tails),
as two, and token by token."""
import numpy as np
import pytest

from workload import synth as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,dk,tail,launches", [(16, 128, 2048, 1), (4, 64, 8192, 1), (16, 128, 1024, 2),
                                                    (4, 64, 4096, 2), (16, 128, 256, 2), (16, 128, 1, 1)])
def test_rounds_in_a_row_carry_the_state(heads, dk, tail, launches):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_18935_gb300 import kvm
    shape = W.ModelShape([W.GDN], 8, 2, 64, 64, 1e4, heads, dk, dk)
    w = W.Workload("back-to-back", 57, shape, [0], 1)
    x = W.device_round_inputs(w, 12, [tail])[0]
    S = torch.from_numpy(W.prefix_state(w, 0, 0)[None]).cuda()
    got = []
    for wait in (True, False):
        ctx = kvm.Context([kvm.LAYER_GDN], 8, 2, 64, 64, 1e4, heads, dk, dk, [64], tail)
        ctx.set_state(0, S)
        outs = [torch.empty((tail, heads, dk), dtype=torch.bfloat16, device="cuda") for _ in range(4)]
        torch.cuda.synchronize()
        before = kvm._lib.kvm_launch_count(ctx._h)
        for out in outs:
            ctx.gdn_chunk_scan_from_state(0, [0, tail], x["q"], x["k"], x["v"], x["alpha"], x["beta"], out)
            if wait:
                torch.cuda.synchronize()
        assert kvm._lib.kvm_launch_count(ctx._h) - before == launches * len(outs)    # the form this size is here for
        got.append([o.view(torch.int16) for o in outs] + [ctx.get_state(0)])
        ctx.check()
    for a, b in zip(*got):
        assert torch.equal(a, b)
