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


def test_runs_by_copies_and_by_pulls():
    """Whole layers arrive as one long run each (copy engine), scattered rows are pulled; both leave the same bytes."""
    L, M, D = 2, 256, 4096     # 24 KB records: 256 adjacent ones are longer than the shortest run that pays a copy
    cfg = synth.StackConfig("runs", L, D, M, 16, 25, 50, 3, 48, 0.9)
    p = Pair(cfg, k=M, C=M, transfer_mode=nb.NP_XFER_MEMCPY_RUNS, staging_rows=200)
    try:
        full = torch.full((L, M // 32), -1, dtype=torch.int32)
        some = synth.random_bitmaps(L, M, 90, 9, 1, 0.5)[0]
        for words, warn in ((full, nb.NP_W_CHUNKED), (some, nb.NP_OK), (full, nb.NP_OK)):
            nb.np_delta(p.eng.ctx, words.cuda(), p.eng.stream)
            assert nb.np_install(p.eng.ctx, 0, L, p.eng.copy_stream) == warn
            p.check_resident_bytes()
            p.check_delta_against(p.ora.res.delta(words.numpy().view(np.uint32)))
    finally:
        p.close()
