"""The kernel that pulls incoming rows from the pinned store: record sizes around its pieces and lines, against the bytes."""
import numpy as np
import pytest
import torch

from paper_2608_22643_b200 import binding as nb
from paper_2608_22643_b200 import synth
from tests.harness import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,records", [
    (8, nb.NP_REC_BF16),       # 48-byte records: a few lanes, any place in a line
    (264, nb.NP_REC_BF16),     # 99 units, one piece
    (1024, nb.NP_REC_BF16),    # 384 units: exactly a piece
    (1536, nb.NP_REC_BF16),    # 576: the last size of one piece and a half
    (1544, nb.NP_REC_BF16),    # 579 units, two pieces, records that start anywhere in a line
    (4104, nb.NP_REC_BF16),    # four pieces, the last one longer
    (16, nb.NP_REC_INT8),      # 64-byte records
    (2048, nb.NP_REC_INT8),    # 384 units and the scales
    (4112, nb.NP_REC_INT8),    # two pieces, the last one longer
])
@pytest.mark.parametrize("mode", [nb.NP_XFER_HOST_GATHER, nb.NP_XFER_ZERO_COPY])
def test_record_sizes(D, records, mode):
    L, M, k = 11, 160, 40      # several launches of uneven shares where the rows are large
    cfg = synth.StackConfig("pull", L, D, M, 16, 25, 50, 4, 47, 0.9)
    p = Pair(cfg, k=k, C=64, transfer_mode=mode, record_format=records, store_layers=3)
    try:
        words = synth.random_bitmaps(L, M, k, 9, 4, 0.6)
        for t in range(4):
            nb.np_delta(p.eng.ctx, words[t].cuda(), p.eng.stream)
            nb.np_install(p.eng.ctx, 0, 4, p.eng.copy_stream)
            nb.np_install(p.eng.ctx, 4, L, p.eng.copy_stream)
            p.check_resident_bytes()
            p.check_delta_against(p.ora.res.delta(words[t].numpy().view(np.uint32)))
    finally:
        p.close()


@pytest.mark.parametrize("records,M,staging_rows", [
    (nb.NP_REC_BF16, 256, 200),    # 24 KB records: 256 adjacent ones are longer than the shortest run that pays a copy
    (nb.NP_REC_BF16, 256, 60),     # five chunks a layer
    (nb.NP_REC_INT8, 512, 512),    # 12 KB records, a chunk a layer
    (nb.NP_REC_INT8, 512, 150),    # four
])
def test_runs_by_copies_and_by_pulls(records, M, staging_rows):
    """Whole layers arrive as one long run each (copy engine), scattered rows are pulled; both leave the same bytes."""
    L, D = 2, 4096
    cfg = synth.StackConfig("runs", L, D, M, 16, 25, 50, 3, 48, 0.9)
    p = Pair(cfg, k=M, C=M, transfer_mode=nb.NP_XFER_MEMCPY_RUNS, staging_rows=staging_rows, record_format=records)
    try:
        full = torch.full((L, M // 32), -1, dtype=torch.int32)
        none = torch.zeros((L, M // 32), dtype=torch.int32)
        some = synth.random_bitmaps(L, M, min(90, staging_rows), 9, 1, 0.5)[0]
        chunked = nb.NP_W_CHUNKED if M > staging_rows else nb.NP_OK
        rest = nb.NP_W_CHUNKED if M - min(90, staging_rows) > staging_rows else nb.NP_OK
        for words, warn, scatters in ((full, chunked, True), (some, nb.NP_OK, False), (full, rest, False), (none, nb.NP_OK, False),
                                      (some, nb.NP_OK, False), (none, nb.NP_OK, False), (full, chunked, True)):
            nb.np_delta(p.eng.ctx, words.cuda(), p.eng.stream)
            before = nb.np_launch_count(p.eng.ctx)
            assert nb.np_install(p.eng.ctx, 0, L, p.eng.copy_stream) == warn
            # a scatter kernel per chunk of a layer behind its copies
            if scatters:
                assert nb.np_launch_count(p.eng.ctx) - before == L * -(-M // staging_rows)
            p.check_resident_bytes()
            p.check_delta_against(p.ora.res.delta(words.numpy().view(np.uint32)))
    finally:
        p.close()


@pytest.mark.parametrize("records", [nb.NP_REC_BF16, nb.NP_REC_INT8])
@pytest.mark.parametrize("staging_rows", [None, 2, 9])
def test_packed_records_in_chunks(records, staging_rows):
    """Host threads pack the records into parts of the pinned staging however few rows a part holds."""
    cfg = synth.CONFIGS["small"]
    p = Pair(cfg, transfer_mode=nb.NP_XFER_HOST_GATHER, staging_rows=staging_rows, record_format=records,
             flags=nb.NP_F_CHECK_BOUNDS | nb.NP_F_MAPPED_STAGING)
    try:
        words = synth.random_bitmaps(cfg.n_layers, cfg.d_ffn, p.k, 5, 4, 0.8)
        words[:, :, 3] = -1                       # adjacent records
        for t in range(4):
            nb.np_delta(p.eng.ctx, words[t].cuda(), p.eng.stream)
            rc = nb.np_install(p.eng.ctx, 0, cfg.n_layers, p.eng.copy_stream)
            if staging_rows is not None and t == 0:
                assert rc == nb.NP_W_CHUNKED
            p.check_resident_bytes()
            p.check_delta_against(p.ora.res.delta(words[t].numpy().view(np.uint32)))
    finally:
        p.close()
