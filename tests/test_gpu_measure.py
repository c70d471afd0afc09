"""The stand-alone measurement kernel at the edges of its row groups, row widths and storage formats
(needs a GB300).  A block takes 4 to 32 rows depending on the row count, rows are read in 32-byte
pieces with a masked last piece, and FP16 and E4M3 rows are held in registers up to 512 entries and read
twice beyond.  Conditionals of every row are compared with the FP64 oracle at the tolerance of the path."""
import numpy as np
import pytest

import gen
import parity
from oracle import quant

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "bf16x2": 1e-4, "bf16x3l": 1e-4, "fp16x2": 1e-4}


def _stored(ts, precision):
    if precision == "fp32":
        return ts
    return [quant.dequant_fp16(A, 1) if precision == "fp16x2" else quant.dequant_bf16(A, 1) for A in ts]


@pytest.mark.parametrize("precision", ["fp32", "bf16x2", "bf16x3l", "fp16x2"])
@pytest.mark.parametrize("d,bonds", [
    (3, [1, 3, 1, 2, 6, 17, 33, 15, 5, 2, 1]),                # odd and one-entry blocks, next rows of 64 entries
    (10, [1, 10, 100, 1050, 105, 11, 2, 1]),                  # rows of many pieces
    (255, [1, 3, 20, 1]),                                     # the most outcomes a site may have
])
def test_measure_edges_against_oracle(precision, d, bonds):
    import paper_2512_20064_gb300 as F

    b, ts, _ = gen.mps_tensors(len(bonds) - 1, d, max(bonds), base_seed=5, skew=1.5 if d < 255 else None,
                               dtype=np.complex64, bonds=bonds)
    N = 37
    with F.Sampler(precision=precision) as s:
        s.load_chain(ts)
        smp, lp, tr = s.sample(b, d, N, 19, trace_rows=N)
    rep = parity.check(b, _stored(ts, precision), 19, np.arange(N), smp, lp, TOL[precision], dev_trace=tr,
                       trace_rows=N)
    assert rep["prob_rows"] == N


@pytest.mark.parametrize("precision,chi", [("fp32", 27), ("bf16x2", 27), ("fp16x2", 27), ("fp8x2", 27), ("fp32", 90)])
def test_row_groups_give_the_same_bits(precision, chi):
    """A row's result is the same bits in a call of 12000 rows (32 per block of the measurement, 128-row
    tiles of the FP32 contraction) and in calls of 1 to 6000 (fewer rows per block, 64- and 32-row tiles)."""
    import paper_2512_20064_gb300 as F

    b, ts, _ = gen.mps_tensors(10, 3, chi, base_seed=3, skew=1.5, dtype=np.complex64)
    with F.Sampler(precision=precision) as s:
        s.load_chain(ts)
        smp, lp = s.sample(b, 3, 12000, 4)
        for n0, N in ((0, 1), (11, 129), (100, 1300), (5, 2600), (1000, 6000)):
            a, l = s.sample(b, 3, N, 4, n0=n0)
            assert np.array_equal(a, smp[n0:n0 + N]) and np.array_equal(l, lp[n0:n0 + N])


@pytest.mark.parametrize("precision", ["bf16x2", "bf16x3l"])
def test_batched_measurements_at_their_edges(precision):
    """32-row measurements of the batched kernel: row counts around a measurement and an m-tile, chunks of 128
    rows, and d = 40, whose sums do not fit shared memory.  Bit for bit the jobs sampled alone."""
    import paper_2512_20064_gb300 as F

    shapes = [(2, 20, 1), (3, 33, 31), (40, 21, 33), (4, 65, 127), (2, 9, 129), (40, 5, 300)]
    samplers, jobs = [], []
    for j, (d, chi, N) in enumerate(shapes):
        b, ts, _ = gen.mps_tensors(7, d, chi, base_seed=60 + j, skew=1.5 if d < 40 else None, dtype=np.complex64)
        s = F.Sampler(precision=precision)
        s.load_chain(ts)
        samplers.append(s)
        jobs.append(dict(chain=s.h, bonds=b, d=d, N=N, seed=5 + j, job=j, n0=3 * j,
                         out_samples=np.empty((N, 7), np.uint8), out_logprob=np.empty(N, np.float64)))
    with F.Sampler(precision=precision, max_microbatch=128) as runner:
        F.fastmps_sample_batch(runner.h, jobs)
    for s, j in zip(samplers, jobs):
        a, l = s.sample(j["bonds"], j["d"], j["N"], j["seed"], n0=j["n0"], job=j["job"])
        assert np.array_equal(a, j["out_samples"]) and np.array_equal(l, j["out_logprob"])
        s.close()


@pytest.mark.parametrize("precision,d,chi", [("bf16x2", 4, 20), ("fp32", 4, 17), ("bf16x2", 3, 700), ("fp32", 9, 12),
                                             ("bf16x2", 8, 256), ("fp32", 16, 6)])
def test_displaced_micro_batches_give_the_same_bits(precision, d, chi):
    """Displaced rows in one micro-batch per site (one stream; matrices and logarithms beside the contraction) and
    in several (two streams), for each variant of the measurement: bit for bit the same, and within tolerance of
    the oracle."""
    import paper_2512_20064_gb300 as F

    M, N = 6, 300
    b, ts, _ = gen.mps_tensors(M, d, chi, base_seed=15, skew=1.5, dtype=np.complex64)
    mu = gen.gbs_amplitudes(M, N, 0.4, seed=8)
    out = []
    for mb in (0, 128):
        with F.Sampler(precision=precision, max_microbatch=mb) as s:
            s.load_chain(ts)
            for _ in range(2):  # a second call finds the buffers of the first
                out.append(s.sample(b, d, N, 6, mu=mu, trace_rows=N))
    for o in out[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(out[0], o))
    smp, lp, tr = out[0]
    parity.check(b, _stored(ts, precision), 6, np.arange(N), smp, lp, TOL[precision], dev_trace=tr, trace_rows=N, mu=mu)


@pytest.mark.parametrize("d", [2, 4, 5, 8])
def test_displacement_pairs_and_singles_give_the_same_bits(d):
    """Two samples per thread (even counts, aligned arrays) against one (odd counts, 8-byte aligned arrays)."""
    import torch

    import paper_2512_20064_gb300 as F

    mu = torch.from_numpy(gen.gbs_amplitudes(1, 771, 0.6, seed=3)[0]).cuda()
    with F.Sampler() as s:
        ref = s.displacement(mu, d)  # 771: singles
        for n in (1, 2, 512, 770):
            assert np.array_equal(s.displacement(mu[:n], d), ref[:, :, :n])
            shifted = torch.empty(d * d * n + 1, dtype=torch.complex64, device="cuda")[1:]
            F.fastmps_displacement(s.h, mu[:n], d, out=shifted)
            assert np.array_equal(shifted.cpu().numpy().reshape(d, d, n), ref[:, :, :n])


@pytest.mark.parametrize("precision", ["fp16x2", "fp16x3", "bf16x2"])
def test_rows_around_the_piece_that_stays_in_registers(precision):
    """Next rows of 512 entries, the widest that a warp scales without a second read, and of 576 (FP16); pieces of
    eight entries whose last one holds 2, 4 or 6 real ones."""
    import paper_2512_20064_gb300 as F

    bonds = [1, 10, 100, 255, 256, 257, 256, 255, 97, 10, 1]
    b, ts, _ = gen.mps_tensors(len(bonds) - 1, 10, 257, base_seed=12, skew=1.5, dtype=np.complex64, bonds=bonds)
    stored = [quant.dequant_fp16(A, 2) for A in ts] if precision == "fp16x3" else _stored(ts, precision)
    N = 41
    with F.Sampler(precision=precision) as s:
        s.load_chain(ts)
        smp, lp, tr = s.sample(b, 10, N, 29, trace_rows=N)
    parity.check(b, stored, 29, np.arange(N), smp, lp, 1e-4, dev_trace=tr, trace_rows=N)


def test_small_fp32_chain_on_the_measurement_kernel():
    """Odd and one-entry blocks of a chain that runs in one launch by itself, in micro-batches of 128 rows: the
    stand-alone measurement kernel against the oracle."""
    import paper_2512_20064_gb300 as F

    bonds = [1, 3, 1, 2, 6, 17, 33, 15, 5, 2, 1]
    b, ts, _ = gen.mps_tensors(len(bonds) - 1, 3, 33, base_seed=5, skew=1.5, dtype=np.complex64, bonds=bonds)
    N = 300
    with F.Sampler(precision="fp32", max_microbatch=128) as s:
        s.load_chain(ts)
        smp, lp, tr = s.sample(b, 3, N, 19, trace_rows=N)
        assert s.stats()["contract_launches"] == 3 * len(ts)
    parity.check(b, ts, 19, np.arange(N), smp, lp, TOL["fp32"], dev_trace=tr, trace_rows=N)
