"""What a step promises about the caller's streams: the order of its rows with the caller's own work."""
import numpy as np
import pytest
import torch

from oracle import np_oracle as O
from paper_2608_22643_b200 import binding as nb
from paper_2608_22643_b200 import synth
from tests.harness import Pair, rel_l2

pytestmark = pytest.mark.gpu

TINY = synth.CONFIGS["tiny"]      # one launch pulls the rows of a step
SMALL = synth.CONFIGS["small"]
MANY = synth.StackConfig("many", 12, 1024, 2048, 64, 30, 60, 4, 51, 0.9)   # several launches on copy_stream

DELAY = 20_000_000                # cycles of a bounded device-side sleep, about 10 ms; a step of these stacks takes 0.1


@pytest.mark.parametrize("mode", [nb.NP_XFER_MEMCPY_RUNS, nb.NP_XFER_HOST_GATHER, nb.NP_XFER_ZERO_COPY])
@pytest.mark.parametrize("cfg", [TINY, SMALL, MANY])
def test_rows_wait_for_what_copy_stream_holds(cfg, mode):
    """A write to the store that copy_stream holds when a step is queued is seen by its rows; a copy of the row buffers
    that copy_stream holds sees the rows of the step before."""
    p = Pair(cfg, transfer_mode=mode)
    try:
        e = p.eng
        words = synth.random_bitmaps(cfg.n_layers, cfg.d_ffn, p.k, 5, 4, 0.5)
        x = synth.hidden_states(cfg, 1)[0].cuda()
        out = torch.empty((1, cfg.d_model), dtype=torch.float32, device="cuda")
        fresh = torch.randn(p.backing.shape, generator=torch.Generator().manual_seed(3)).to(torch.bfloat16).cuda()
        snap = torch.empty_like(e.gate)
        for t in range(4):
            before = e.gate.clone()
            torch.cuda.synchronize()
            with torch.cuda.stream(e.copy_stream):
                torch.cuda._sleep(DELAY)
                snap.copy_(e.gate)
                if t == 2:
                    p.backing.copy_(fresh, non_blocking=True)
            assert not e.copy_stream.query()
            nb.np_step_selected(e.ctx, x, 1, words[t].cuda(), out, e.stream, e.copy_stream)
            after = torch.empty_like(e.gate)
            with torch.cuda.stream(e.copy_stream):      # queued behind the step: sees its rows
                after.copy_(e.gate)
            torch.cuda.synchronize()
            assert torch.equal(snap, before), t
            assert torch.equal(after, e.gate), t
            if t == 2:                                   # every row of this step is one of the new records
                c = e.counters()
                for l in range(cfg.n_layers):
                    d = e.delta_lists(l, c[l])
                    assert len(d["delta_ids"]) > 0
                    want = fresh[l, torch.from_numpy(d["delta_ids"].copy()).cuda().long()]
                    for i, buf in enumerate((e.gate, e.up, e.downT)):
                        assert torch.equal(buf[l, torch.from_numpy(d["delta_slots"].copy()).cuda().long()], want[:, i]), (l, i)
    finally:
        p.close()


@pytest.mark.parametrize("second", ["last layer", "speculative"])
def test_marks_survive_an_install_on_another_stream(second):
    """A layer's MLP waits for its rows on one stream also after another install has marked that layer, or the last
    layer of its launch, on a second stream."""
    cfg = SMALL
    p = Pair(cfg, transfer_mode=nb.NP_XFER_ZERO_COPY)
    try:
        e, L, D = p.eng, cfg.n_layers, cfg.d_model
        other = torch.cuda.Stream()
        words = synth.random_bitmaps(L, cfg.d_ffn, p.k, 5, 3, 0.3)
        x = np.random.default_rng(8).standard_normal((1, D)).astype(np.float32)
        xd = torch.from_numpy(x).cuda()
        y = torch.empty((L, 1, D), dtype=torch.float32, device="cuda")
        for t in range(3):
            nb.np_delta(e.ctx, words[t].cuda(), e.stream)
            torch.cuda.synchronize()
            with torch.cuda.stream(e.copy_stream):
                torch.cuda._sleep(DELAY)
            nb.np_install(e.ctx, 0, L, e.copy_stream)
            if second == "speculative":
                nb.np_speculate(e.ctx, words[(t + 1) % 3].cuda(), 8, e.stream)
                nb.np_install_speculative(e.ctx, other)
            else:
                nb.np_install(e.ctx, L - 1, L, other)
            for l in range(L):
                nb.np_sparse_mlp(e.ctx, l, xd, 1, y[l], e.stream)
            torch.cuda.synchronize()
            deltas = p.ora.res.delta(words[t].numpy().view(np.uint32))
            for l, d in enumerate(deltas):
                O.install(p.store_u16, p.ora.gate, p.ora.up, p.ora.downT, l, d.delta_ids, d.delta_slots)
                want = O.sparse_mlp(p.ora.gate, p.ora.up, p.ora.downT, l, d.active_slots, x.astype(np.float64))
                assert rel_l2(y[l].cpu().numpy(), want) < 1e-5, (t, l)    # fp32 sums of bf16 products: 1e-6
            if second == "speculative":
                break                          # the oracle above holds no speculative rows
    finally:
        p.close()


@pytest.mark.parametrize("cfg", [TINY, MANY])
def test_step_times_are_those_of_the_step(cfg):
    """np_last_step_times after other calls, one of them not finished, reports what it reported right behind the step, and
    waits for no work of the program's own."""
    p = Pair(cfg, with_oracle=False)
    try:
        e = p.eng
        words = synth.random_bitmaps(cfg.n_layers, cfg.d_ffn, p.k, 5, 4, 0.5)
        x = synth.hidden_states(cfg, 1)[0].cuda()
        out = torch.empty((1, cfg.d_model), dtype=torch.float32, device="cuda")
        later = words[1:].cuda()
        for t in range(3):
            nb.np_step(e.ctx, x, 1, out, e.stream, e.copy_stream)
            first = nb.np_last_step_times(e.ctx)
            assert (first > 0).all(), t
            nb.np_delta(e.ctx, words[t].cuda(), e.stream)
            nb.np_install(e.ctx, 0, cfg.n_layers, e.copy_stream)
            assert (nb.np_last_step_times(e.ctx) == first).all(), t
            torch.cuda.synchronize()
            torch.cuda._sleep(10 * DELAY)
            with torch.cuda.stream(e.stream):
                torch.cuda._sleep(DELAY)
            nb.np_delta(e.ctx, later[t], e.stream)
            assert (nb.np_last_step_times(e.ctx) == first).all(), t
            assert not torch.cuda.default_stream().query() and not e.stream.query(), t
            torch.cuda.synchronize()
            nb.np_install(e.ctx, 0, cfg.n_layers, e.copy_stream)
    finally:
        p.close()
