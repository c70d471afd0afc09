"""Row counts that end inside an m-tile, or leave a pair of thread blocks with one m-tile only, and calls on pairs
against calls on single blocks (needs a GB300).  A row's result depends on no other row, so it has the same bits
whatever the row count, the micro-batch or the kind of launch.

A warp of the contraction whose 32 rows lie past the last one stores nothing, but keeps its place among the staging
buffers of the scratch stores: at these counts a block goes from tiles with rows to tiles without."""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu

M, D = 12, 4
FULL = 41 * 256  # rows: 82 whole m-tiles


def _chain(chi):
    b, ts, _ = gen.mps_tensors(M, D, chi, base_seed=500 + chi, skew=1.5, dtype=np.complex64)
    return b, ts


@pytest.mark.parametrize("precision,chunk,chi", [
    ("bf16x2", 0, 256),  # pairs, 8 column tiles of 256: 41 x 8 units of two m-tiles on 76 pairs
    ("bf16x3", 0, 200),  # pairs, two site planes
    ("bf16x2", 0, 64),   # pairs, column tiles of 128
    ("bf16x2", 0, 80),   # pairs, column tiles of 160: half a tile is 80
    ("fp16x3", 0, 100),  # pairs, FP16
    ("bf16x2", 0, 40),   # single blocks, column tiles of 96 (three chunks of 32): 82 x 4 tiles on 152 SMs
    ("bf16x3l", 0, 24),  # single blocks, column tiles of 64
    ("bf16x2", 0, 16),   # single blocks, column tiles of 32: one chunk
    ("fp16x2", 4, 200),  # pairs, promoted accumulation
    ("fp8x2", 0, 100),   # single blocks, FP8
])
def test_rows_past_the_last_one_change_no_bits(precision, chunk, chi):
    import paper_2512_20064_gb300 as F

    b, ts = _chain(chi)
    with F.Sampler(precision=precision, accum_chunk=chunk) as s:
        s.load_chain(ts)
        smp, lp = s.sample(b, D, FULL, 31)
        for r in (1, 33, 65, 97, 129):
            a, l = s.sample(b, D, FULL - 256 + r, 31)
            assert np.array_equal(a, smp[:len(a)]) and np.array_equal(l, lp[:len(a)]), r


@pytest.mark.parametrize("precision,chunk,chi", [("bf16x2", 0, 256), ("bf16x3", 0, 64), ("fp16x2", 4, 200)])
def test_micro_batch_that_ends_inside_a_pair(precision, chunk, chi):
    """Nine m-tiles per micro-batch: the last pair's second block has none."""
    import paper_2512_20064_gb300 as F

    b, ts = _chain(chi)
    out = []
    for mb in (0, 9 * 128):
        with F.Sampler(precision=precision, accum_chunk=chunk, max_microbatch=mb) as s:
            s.load_chain(ts)
            out.append(s.sample(b, D, FULL - 95, 8, trace_rows=300))
    assert all(np.array_equal(x, y) for x, y in zip(*out))


@pytest.mark.parametrize("precision,chi", [("bf16x2", 256), ("bf16x3", 200), ("bf16x3l", 64), ("bf16x4", 80)])
def test_pairs_equal_single_blocks(precision, chi):
    """fastmps_sample_noalloc never launches pairs."""
    import torch

    import paper_2512_20064_gb300 as F

    b, ts = _chain(chi)
    with F.Sampler(precision=precision) as s:
        s.load_chain(ts)
        for N in (129, 257, 1500):  # 2, 3 and 12 m-tiles
            a, l = s.sample(b, D, N, 3)
            o = torch.empty((N, M), dtype=torch.uint8, device="cuda")
            p = torch.empty(N, dtype=torch.float64, device="cuda")
            F.fastmps_sample_noalloc(s.h, M, D, b, 0, N, 3, 0, o, p)
            assert np.array_equal(a, o.cpu().numpy()) and np.array_equal(l, p.cpu().numpy()), N
