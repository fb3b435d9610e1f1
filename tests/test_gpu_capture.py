"""Calls that queue device work only may be captured into a graph, and the graph replayed on new contents of its buffers."""
import numpy as np
import pytest
import torch

from oracle import np_oracle as O
from paper_2608_22643_b200 import binding as nb
from paper_2608_22643_b200 import synth
from tests.harness import Pair, rel_l2, u16

pytestmark = pytest.mark.gpu

TOL = 1e-5    # fp32 sums of bf16 products: 1e-6


def _stack(D):
    return synth.StackConfig("cap", 3, D, 1024, 64, 25, 50, 4, 29, 0.9)


@pytest.mark.parametrize("D,B,dense,flags", [
    (256, 1, 0, 0), (272, 1, 0, 0), (264, 1, 0, 0),       # the sliced kernel, even and uneven; a width it does not take
    (256, 1, 0, nb.NP_F_CLUSTER_ROWS), (1024, 1, 0, nb.NP_F_CLUSTER_ROWS), (256, 1, 1, 0),
    (256, 4, 0, 0), (272, 3, 0, 0), (256, 16, 0, 0), (256, 4, 1, 0), (256, 4, 0, nb.NP_F_TCGEN05_BATCH),
])
def test_chain_replays(D, B, dense, flags):
    """The graph's chain gives what the call gives, replay after replay, with calls in between."""
    cfg = _stack(D)
    p = Pair(cfg, max_batch=B, C=1024, dense_layers=dense, flags=flags | nb.NP_F_CHECK_BOUNDS, with_oracle=False)
    try:
        e = p.eng
        xs = synth.hidden_states(cfg, 4, batch=B)
        x = xs[0].cuda()
        out, again = (torch.empty((B, D), dtype=torch.float32, device="cuda") for _ in range(2))
        nb.np_step(e.ctx, x, B, out, e.stream, e.copy_stream)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=e.stream):
            nb.np_mlp_chain(e.ctx, x, B, out, e.stream)
        for t in range(4):
            x.copy_(xs[t])
            torch.cuda.synchronize()
            out.fill_(float("nan"))
            g.replay()
            torch.cuda.synchronize()
            nb.np_mlp_chain(e.ctx, x, B, again, e.stream)
            e.counters()
            assert rel_l2(out.cpu().numpy(), again.cpu().numpy()) < TOL, t
    finally:
        p.close()


@pytest.mark.parametrize("B", [1, 4])
def test_delta_install_and_mlp_replay(B):
    """Selection by the caller, delta, install without the host and the layers' MLP in one graph over two streams."""
    cfg = _stack(256)
    L, D = cfg.n_layers, cfg.d_model
    p = Pair(cfg, max_batch=B, transfer_mode=nb.NP_XFER_ZERO_COPY)
    try:
        e = p.eng
        words = synth.random_bitmaps(L, cfg.d_ffn, p.k, 5, 5, 0.6)
        sel = words[0].cuda()
        x = np.random.default_rng(3).standard_normal((B, D)).astype(np.float32)
        xd = torch.from_numpy(x).cuda()
        y = torch.empty((L, B, D), dtype=torch.float32, device="cuda")
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=e.stream):
            nb.np_delta(e.ctx, sel, e.stream)
            nb.np_install(e.ctx, 0, L, e.copy_stream)
            for l in range(L):
                nb.np_sparse_mlp(e.ctx, l, xd, B, y[l], e.stream)
        for t in range(5):
            sel.copy_(words[t])
            torch.cuda.synchronize()
            y.fill_(float("nan"))
            g.replay()
            torch.cuda.synchronize()
            e.counters()
            for l, d in enumerate(p.ora.res.delta(words[t].numpy().view(np.uint32))):
                O.install(p.store_u16, p.ora.gate, p.ora.up, p.ora.downT, l, d.delta_ids, d.delta_slots)
                want = O.sparse_mlp(p.ora.gate, p.ora.up, p.ora.downT, l, d.active_slots, x.astype(np.float64))
                assert rel_l2(y[l].cpu().numpy(), want) < TOL, (t, l)
            p.check_resident_bytes()
    finally:
        p.close()


@pytest.mark.parametrize("B", [1, 5])
def test_predict_replays(B):
    cfg = _stack(256)
    L, M = cfg.n_layers, cfg.d_ffn
    p = Pair(cfg, max_batch=B, C=M, with_oracle=False)
    try:
        xs = synth.hidden_states(cfg, 3, batch=B)
        x = xs[0].cuda()
        logits = torch.empty((B, L, M), dtype=torch.float32, device="cuda")
        words = torch.empty((L, M // 32), dtype=torch.int32, device="cuda")
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=p.eng.stream):
            nb.np_predict(p.eng.ctx, x, B, logits, words, p.eng.stream)
        for t in range(3):
            x.copy_(xs[t])
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            z = O.predict(u16(p.w1_cpu), u16(p.w2_cpu), u16(xs[t]), L, M)
            assert rel_l2(logits.cpu().numpy(), z) < TOL, t
            assert (words.cpu().numpy().view(np.uint32) == O.topk_bitmap(logits.cpu().numpy(), p.k)).all(), t
    finally:
        p.close()
