"""Launches whose dynamic shared memory fits 48 KB by itself but not beside the kernel's own variables."""
import pytest
import torch

from paper_2608_22643_b200 import binding as nb
from paper_2608_22643_b200 import synth
from tests.harness import Pair, rel_l2, u16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,C", [(6144, 2208), (6144, 2240), (6144, 2457), (6144, 3328), (6144, 3329), (5504, 5504), (6976, 37)])
def test_delta(M, C):
    """32 (M / 32) + 8 (C / 32) bytes beside 42176: 48880 to 49152 of them, and the sizes around."""
    cfg = synth.StackConfig("smem", 2, 64, M, 16, 1, 2, 3, 29, 0.9)
    p = Pair(cfg, k=min(C, 300), C=C)
    try:
        xs = synth.hidden_states(cfg, 3)
        out = torch.empty((1, 64), dtype=torch.float32, device="cuda")
        logits = torch.empty((1, 2, M), dtype=torch.float32, device="cuda")
        for t in range(3):
            nb.np_predict(p.eng.ctx, xs[t].cuda(), 1, logits, None, p.eng.stream)
            nb.np_step(p.eng.ctx, xs[t].cuda(), 1, out, p.eng.stream, p.eng.copy_stream)
            torch.cuda.synchronize()
            p.check_delta_against(p.ora.step(u16(xs[t]), logits_f32=logits.cpu().numpy())["deltas"])
    finally:
        p.close()


@pytest.mark.parametrize("D,B", [(2520, 4), (2528, 4), (2536, 4), (2544, 4), (2552, 4), (5600, 2), (5616, 2), (5624, 2), (11744, 1), (11760, 1), (11768, 1)])
def test_mlp_with_direct_loads(D, B):
    """4 B (D + 528) bytes for up to four sequences."""
    M, k = 64, 20
    cfg = synth.StackConfig("smem", 1, D, M, 16, 1, 2, 1, 31, 0.9)
    p = Pair(cfg, max_batch=B, k=k, C=M, flags=nb.NP_F_CHECK_BOUNDS | nb.NP_F_DIRECT_LOADS)
    try:
        x = synth.hidden_states(cfg, 1, batch=B)[0]
        logits = torch.empty((B, 1, M), dtype=torch.float32, device="cuda")
        out = torch.empty((B, D), dtype=torch.float32, device="cuda")
        nb.np_predict(p.eng.ctx, x.cuda(), B, logits, None, p.eng.stream)
        nb.np_step(p.eng.ctx, x.cuda(), B, out, p.eng.stream, p.eng.copy_stream)
        torch.cuda.synchronize()
        want = p.ora.step(u16(x), logits_f32=logits.cpu().numpy())["x_final"]
        for b in range(B):
            assert rel_l2(out.cpu().numpy()[b], want[b]) < 1e-5, b   # fp32 sums of bf16 products: 1e-6
    finally:
        p.close()
