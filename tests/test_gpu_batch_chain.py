"""The resident MLP kernel for batches at the edges of its partition, against the oracle."""
import pytest
import torch

from paper_2608_22643_b200 import binding as nb
from paper_2608_22643_b200 import synth
from tests.harness import Pair, rel_l2, u16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,M,k,chain_layers", [
    (16, 64, 5, 0),          # one K block, row groups without rows
    (32, 256, 200, 0),       # two slices of one K block each
    (48, 256, 200, 0),       # three
    (272, 4096, 3000, 0),    # four slices of 4 and 5 K blocks; six chunks of rows per block, ragged
    (1296, 512, 200, 2),     # 20 and 21 K blocks, a launch per two layers
    (2064, 512, 200, 0),     # 32 and 33: a K block more than four per warp, the instance for up to eight
    (2064, 2656, 2600, 0),   # five chunks per block, the last one of 6 or 7 rows
    (4112, 2656, 2600, 1),   # 64 and 65: the instance for up to ten
    (5120, 2656, 2650, 0),   # 80: the widest slice
    (8208, 256, 130, 1),     # eight slices of 64 and 65, a launch per layer
    (24, 64, 9, 0),          # not a multiple of 16: the kernel does not apply
])
@pytest.mark.parametrize("B", [2, 8, 9, 16])
def test_chain_at_partition_edges(D, M, k, chain_layers, B):
    L = 3 if D * M < 5e6 else 2
    cfg = synth.StackConfig("bc", L, D, M, 32, 25, 50, 3, 23, 0.9)
    p = Pair(cfg, max_batch=B, k=k, C=M, chain_layers=chain_layers, gen_device="cuda" if D * M > 5e6 else "cpu")
    try:
        assert (nb.np_mlp_kernel_name(p.eng.ctx, B) == "k_mlp_batch") == (D % 16 == 0)
        xs = synth.hidden_states(cfg, 3, batch=B)
        out = torch.empty((B, D), dtype=torch.float32, device="cuda")
        logits = torch.empty((B, L, M), dtype=torch.float32, device="cuda")
        for t in range(3):
            nb.np_predict(p.eng.ctx, xs[t].cuda(), B, logits, None, p.eng.stream)
            nb.np_step(p.eng.ctx, xs[t].cuda(), B, out, p.eng.stream, p.eng.copy_stream)
            torch.cuda.synchronize()
            res = p.ora.step(u16(xs[t]), logits_f32=logits.cpu().numpy())
            p.check_delta_against(res["deltas"])
            got = out.cpu().numpy()
            for b in range(B):
                assert rel_l2(got[b], res["x_final"][b]) < 1e-5, (t, b)   # fp32 sums of bf16 products: 1e-6
        p.eng.counters()
    finally:
        p.close()
