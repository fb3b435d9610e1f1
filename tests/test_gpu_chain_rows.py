"""The column-sliced MLP kernel where its row groups and its shared memory run out, against the oracle."""
import pytest
import torch

from paper_2608_22643_b200 import binding as nb
from paper_2608_22643_b200 import synth
from tests.harness import Pair, rel_l2, u16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,M,k,L", [
    (256, 4096, 37 * 32, 3),      # a row per lane in every row group of 148 SMs
    (256, 4096, 37 * 32 + 1, 3),  # one row group of 33
    (256, 4096, 37 * 64, 3),
    (256, 4096, 37 * 64 + 1, 3),  # one of 65: a second round of the exchange
    (256, 4096, 4096, 3),
    (1216, 2048, 37 * 39, 3),     # 39 rows, 19 K blocks of a slice
    (4160, 2048, 37 * 39, 2),     # 65 K blocks of a slice: nine for each warp, two for the last
    (80, 512, 130, 3),            # slices of one and two K blocks
    (2384, 4096, 37 * 30, 3),     # slices of 37 and 38
    (4144, 2048, 37 * 39, 2),     # slices of 64 and 65
    (8176, 512, 100, 2),          # the widest slice holds a tile more than the others
    (8192, 8320, 1040, 1),        # a capacity of 8320: the slots of two layers take their part of the shared memory
    (8256, 512, 100, 3),          # the narrowest rows that another kernel takes
])
def test_chain_row_groups(D, M, k, L):
    cfg = synth.StackConfig("rows", L, D, M, 32, 25, 50, 3, 23, 0.9)
    p = Pair(cfg, max_batch=1, k=k, C=M)
    try:
        xs = synth.hidden_states(cfg, 3, batch=1)
        out = torch.empty((1, D), dtype=torch.float32, device="cuda")
        logits = torch.empty((1, L, M), dtype=torch.float32, device="cuda")
        for t in range(3):
            nb.np_predict(p.eng.ctx, xs[t].cuda(), 1, logits, None, p.eng.stream)
            nb.np_step(p.eng.ctx, xs[t].cuda(), 1, out, p.eng.stream, p.eng.copy_stream)
            torch.cuda.synchronize()
            res = p.ora.step(u16(xs[t]), logits_f32=logits.cpu().numpy())
            p.check_delta_against(res["deltas"])
            assert rel_l2(out.cpu().numpy()[0], res["x_final"][0]) < 1e-5, t  # fp32 sums of bf16 products: 1e-6
        p.eng.counters()
    finally:
        p.close()


@pytest.mark.parametrize("D,M,k,L", [
    (64, 512, 60, 130),           # one K block per slice, a single warp; more layers than a launch covers
    (128, 512, 10, 3),            # two K blocks, row groups without rows
    (512, 2048, 37 * 16 + 1, 3),  # a down tile of one row in one row group
    (576, 1024, 100, 3),          # nine K blocks of a slice on five warps of two: a ragged last warp
    (2064, 1024, 37 * 8, 3),      # slices of 32 and 33 K blocks: two and three of five for the last warp
    (5120, 2048, 37 * 48, 2),     # rounds of the exchange of 48 rows: one full
    (5120, 2048, 37 * 48 + 1, 2), # a second round of one row
    (6144, 2560, 37 * 65, 2),     # two rounds of 64 rows, two buffers
    (8192, 2560, 37 * 33, 2),     # one tile held at a time, five to a layer
    (8176, 2048, 37 * 17, 2),     # the same at uneven slices
    # the other instances, each with a ragged number of tiles
    (528, 512, 338, 2),           # one or two K blocks for a warp, the last one without any in three slices
    (640, 512, 338, 2),           # two for each
    (1152, 512, 338, 2),          # three
    (1168, 512, 338, 2),          # three, none for the last warp in three slices
    (1552, 512, 338, 2),          # four, the same
    (2000, 512, 338, 2),          # four, three for the last
    (2048, 512, 338, 2),
    (2256, 512, 338, 2),          # five, none for the last warp in three slices
    (2560, 512, 338, 2),
    (2640, 512, 338, 2),          # six, five for the last
    (2704, 512, 338, 2),          # six, none for the last warp in three slices
    (3072, 512, 338, 2),
    (3152, 512, 338, 2),          # seven where the instance has eight, none for the last warp in three slices
    (3520, 512, 338, 2),          # seven, six for the last
    (4080, 512, 338, 2),          # eight, seven for the last
    (5104, 512, 338, 2),          # ten, nine for the last
    (5488, 512, 338, 2),          # eleven where the instance has twelve
    (6128, 512, 338, 2),          # twelve, eleven for the last
    (6672, 512, 338, 2),          # fourteen where the instance has sixteen, its second half partly filled
    (7184, 512, 338, 2),          # fifteen, seven for the last: its second half is empty
])
def test_chain_tiles(D, M, k, L):
    cfg = synth.StackConfig("tiles", L, D, M, 32, 25, 50, 2, 29, 0.9)
    p = Pair(cfg, max_batch=1, k=k, C=max(k, M // 2))
    try:
        xs = synth.hidden_states(cfg, 2, batch=1)
        out = torch.empty((1, D), dtype=torch.float32, device="cuda")
        logits = torch.empty((1, L, M), dtype=torch.float32, device="cuda")
        for t in range(2):
            x = xs[t].cuda()
            nb.np_predict(p.eng.ctx, x, 1, logits, None, p.eng.stream)
            nb.np_step(p.eng.ctx, x, 1, out, p.eng.stream, p.eng.copy_stream)
            torch.cuda.synchronize()
            res = p.ora.step(u16(xs[t]), logits_f32=logits.cpu().numpy())
            # fp32 sums of bf16 products: 1e-6 over a few layers; layers past 20 add in proportion
            tol = 1e-5 * max(1.0, L / 20)
            assert rel_l2(out.cpu().numpy()[0], res["x_final"][0]) < tol, t
            nb.np_mlp_chain(p.eng.ctx, x, 1, out, p.eng.stream)      # resident rows: one run, as few launches as there can be
            torch.cuda.synchronize()
            assert rel_l2(out.cpu().numpy()[0], res["x_final"][0]) < tol, t
            assert nb.np_chain_launches(p.eng.ctx) == (L + 127) // 128
        p.eng.counters()
    finally:
        p.close()


def test_launches_of_the_row_partitioned_kernel():
    """More layers than one of its launches covers: both are counted."""
    cfg = synth.StackConfig("long", 130, 64, 128, 32, 25, 50, 1, 31, 0.9)
    p = Pair(cfg, max_batch=1, flags=nb.NP_F_CHECK_BOUNDS | nb.NP_F_ROW_CHAIN, with_oracle=False)
    try:
        assert nb.np_mlp_kernel_name(p.eng.ctx, 1) == "k_mlp_chain_alu"
        x = synth.hidden_states(cfg, 1)[0].cuda()
        out = torch.empty((1, cfg.d_model), dtype=torch.float32, device="cuda")
        nb.np_step(p.eng.ctx, x, 1, out, p.eng.stream, p.eng.copy_stream)
        torch.cuda.synchronize()
        nb.np_mlp_chain(p.eng.ctx, x, 1, out, p.eng.stream)
        torch.cuda.synchronize()
        assert nb.np_chain_launches(p.eng.ctx) == 2
        p.eng.counters()
    finally:
        p.close()
