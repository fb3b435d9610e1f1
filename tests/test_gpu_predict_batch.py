"""np_predict for batches on the tensor cores: ragged widths of both layers, and the caller's outputs."""
import numpy as np
import pytest
import torch

from oracle import np_oracle as O
from paper_2608_22643_b200 import binding as nb
from paper_2608_22643_b200 import synth
from tests.harness import Pair, rel_l2, u16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,H", [(8, 8), (72, 64), (1000, 136), (2064, 200), (8192, 128), (8200, 64)])
@pytest.mark.parametrize("B", [2, 5, 16])
def test_ragged_widths_match_the_oracle(D, H, B):
    """K blocks of 64 and row tiles of 128 that end past the matrix, one and many K ranges, a width (8200) whose
    layer 1 is outside the tensor-core kernel; 160 rows of layer 2 = a full tile and a quarter."""
    L, M = 5, 32
    p = Pair(synth.StackConfig("pb", L, D, M, H, 25, 50, 2, 43, 0.9), max_batch=B, with_oracle=False)
    try:
        x = synth.hidden_states(p.cfg, 1, batch=B)[0]
        logits = torch.full((B, L, M), 7.0, dtype=torch.float32, device="cuda")
        nb.np_predict(p.eng.ctx, x.cuda(), B, logits, None, p.eng.stream)
        p.eng.counters()
        z = O.predict(u16(p.w1_cpu), u16(p.w2_cpu), u16(x), L, M)
        assert rel_l2(logits.cpu().numpy(), z) < 1e-5    # fp32 accumulation of at most 8200 products: below 1e-6
    finally:
        p.close()


@pytest.mark.parametrize("B", [1, 2, 16])
@pytest.mark.parametrize("k", [0, 7, 96])
def test_bitmap_handed_out_is_the_one_kept(B, k):
    """The selection writes the caller's words and the context's own, each call anew."""
    L, M = 3, 96
    p = Pair(synth.StackConfig("po", L, 64, M, 72, 25, 50, 4, 44, 0.5), max_batch=B, k=k, C=M, with_oracle=False)
    try:
        xs = synth.hidden_states(p.cfg, 3, batch=B)
        logits = torch.empty((B, L, M), dtype=torch.float32, device="cuda")
        words = torch.full((L, M // 32), -1, dtype=torch.int32, device="cuda")
        for t in range(3):
            nb.np_predict(p.eng.ctx, xs[t].cuda(), B, logits, words, p.eng.stream)
            nb.np_delta(p.eng.ctx, None, p.eng.stream)
            c = p.eng.counters()
            want = O.topk_bitmap(logits.cpu().numpy(), k)
            got = words.cpu().numpy().view(np.uint32)
            assert (got == want).all(), t
            for l in range(L):
                active = p.eng.delta_lists(l, c[l])["active_ids"]
                assert (active == np.flatnonzero(O.bitmap_to_bool(got[l], M))).all(), (t, l)
    finally:
        p.close()


@pytest.mark.parametrize("M,k", [(32, 5), (512, 511), (544, 100), (6144, 600), (6176, 1), (11264, 1100), (14336, 2000), (14368, 2000)])
def test_more_selections_than_sms(M, k):
    """Blocks of 512 threads take a job each where there are more jobs than SMs: row counts around their keys per thread,
    ordinary logits, heavy ties and infinities."""
    L, B = 10, 16
    p = Pair(synth.StackConfig("tk", L, 16, M, 8, 25, 50, 1, 45, 0.5), max_batch=B, k=k, C=M, with_oracle=False)
    try:
        g = torch.Generator().manual_seed(M)
        z = torch.randn((B, L, M), generator=g)
        z[:, 1] = torch.randint(0, 3, (B, M), generator=g).float()      # ties: more keys in the deciding bin than are ranked
        z[:, 2, ::7] = float("inf")
        z[:, 3] = 0.25
        words = torch.full((L, M // 32), -1, dtype=torch.int32, device="cuda")
        nb.np_topk(p.eng.ctx, z.cuda(), B, words, p.eng.stream)
        p.eng.stream.synchronize()
        for l in range(L):
            want = O.topk_bitmap(z[:, l:l + 1].numpy(), k)[0]
            assert (words[l].cpu().numpy().view(np.uint32) == want).all(), l
    finally:
        p.close()


@pytest.mark.parametrize("B", [2, 3, 16])
def test_hidden_values_at_the_end_of_the_range(B):
    """A hidden value beyond the largest bf16, and one that overflowed to infinity: the scores are those of the product in
    64 bits (infinite with the sign of the weight), and the other sequences' scores do not change."""
    L, M, D, H = 2, 64, 128, 64
    p = Pair(synth.StackConfig("pr", L, D, M, H, 25, 50, 2, 46, 0.9), max_batch=B, with_oracle=False)
    try:
        w1, w2 = p.eng.w1.view(H, D), p.eng.w2.view(L * M, H)
        w1[5, 0], w1[5, 1] = 1.0, 1.0
        w1[6, 2] = 4.0
        x = synth.hidden_states(p.cfg, 1, batch=B)[0].cuda()
        plain = x.clone()
        x[0] = 0
        x[0, 0], x[0, 1] = 3.3895e38, 1.0e36          # hidden value 5 is 3.3995e38: finite, and infinite once rounded to bf16
        x[1] = 0
        x[1, 2] = 3.0e38                              # hidden value 6 is 1.2e39: infinite
        got = torch.empty((B, L * M), dtype=torch.float32, device="cuda")
        rest = torch.empty((B, L * M), dtype=torch.float32, device="cuda")
        nb.np_predict(p.eng.ctx, x, B, got, None, p.eng.stream)
        nb.np_predict(p.eng.ctx, plain, B, rest, None, p.eng.stream)
        p.eng.counters()
        hidden = (x[0].double() @ w1.double().T).clamp(min=0)
        assert 3.396e38 < float(hidden[5]) < 3.4e38
        assert rel_l2(got[0].cpu().numpy(), (w2.double() @ hidden).cpu().numpy()) < 1e-5
        assert torch.equal(got[1], torch.sign(w2[:, 6].float()) * float("inf"))
        assert torch.equal(got[2:], rest[2:])
    finally:
        p.close()


@pytest.mark.parametrize("H", [64, 264, 320, 328, 384, 896, 960, 1024])   # 320: the widest with two tiles to a stage
@pytest.mark.parametrize("L,M", [
    (1, 128),       # a block with one tile: the pair's second is missing
    (37, 1024),     # 296 tiles: a pair for each of 148 SMs
    (38, 1024),     # 304: pairs, and pairs with a tile behind them
    (37, 1056),     # 305.25: the last tile is a quarter
    (75, 1024),     # 600: two pairs and an odd tile on some SMs
])
def test_pairs_of_row_tiles(L, M, H):
    B = 3
    p = Pair(synth.StackConfig("pt", L, 64, M, H, 25, 50, 1, 47, 0.9), max_batch=B, k=1, C=32, with_oracle=False, store_layers=1,
             gen_device="cuda")
    try:
        x = synth.hidden_states(p.cfg, 1, batch=B)[0]
        logits = torch.full((B, L, M), 7.0, dtype=torch.float32, device="cuda")
        nb.np_predict(p.eng.ctx, x.cuda(), B, logits, None, p.eng.stream)
        p.eng.counters()
        z = O.predict(u16(p.w1_cpu), u16(p.w2_cpu), u16(x), L, M)
        assert rel_l2(logits.cpu().numpy(), z) < 1e-5    # fp32 accumulation of at most 1024 products: below 1e-6
    finally:
        p.close()
