"""FP32 calls that run a whole chain in one launch (needs a GB300): bit for bit the results of the two-kernel
path, which fastmps_sample_noalloc takes for every call, and within tolerance of the FP64 oracle.  Widths lie
around the edges of the kernel's units (outcome blocks of 16, 32 and 64 columns side by side, tiles of 64 and
128), chains around the 32 sites whose logarithms are taken together, row counts around a block's 32 rows."""
import numpy as np
import pytest

import gen
import parity

pytestmark = pytest.mark.gpu

CHAINS = [
    (2, [1, 1]),                                               # one site
    (3, [1, 3, 8, 9, 16, 17, 32, 33, 17, 8, 3, 1]),            # 2 chi around 16, 32, 64
    (2, [1, 2, 4, 8, 16, 31, 32, 33, 64, 65, 64, 33, 32, 16, 8, 4, 2, 1]),
    (3, [1, 3, 7, 15, 40, 100, 70, 64, 31, 11, 4, 2, 1]),      # several tiles per outcome, the last one half
    (11, [1, 11, 12, 5, 1]),                                   # outcome blocks that do not fill the last unit
    (60, [1, 2, 1]),
    (2, [1, 2] + [4] * 31 + [2, 1]),                           # 34 sites
]


@pytest.mark.parametrize("d,bonds", CHAINS)
def test_one_launch_equals_two_kernels_and_oracle(d, bonds):
    import torch

    import paper_2512_20064_gb300 as F

    M = len(bonds) - 1
    b, ts, _ = gen.mps_tensors(M, d, max(bonds), base_seed=41, skew=2.0 if d < 60 else None, dtype=np.complex64,
                               bonds=bonds)
    with F.Sampler(precision="fp32") as s:
        s.load_chain(ts)
        for n0, N in ((0, 1), (5, 31), (0, 33), (7, 500)):
            smp, lp = s.sample(b, d, N, 23, n0=n0)
            assert s.stats()["launches"] == 1
            o = torch.empty((N, M), dtype=torch.uint8, device="cuda")
            l = torch.empty(N, dtype=torch.float64, device="cuda")
            F.fastmps_sample_noalloc(s.h, M, d, b, n0, N, 23, 0, o, l)
            assert np.array_equal(smp, o.cpu().numpy()) and np.array_equal(lp, l.cpu().numpy())
        N = 70
        smp, lp, tr = s.sample(b, d, N, 23, trace_rows=N)
        rows = [69, 0, 33]
        smp2, lp2, tr2 = s.sample(b, d, N, 23, trace_list=rows)
        assert np.array_equal(smp, smp2) and np.array_equal(lp, lp2) and np.array_equal(tr[:, rows], tr2)
    rep = parity.check(b, ts, 23, np.arange(N), smp, lp, 1e-5, dev_trace=tr, trace_rows=N)
    assert rep["prob_rows"] == N


def test_one_launch_reports_a_zero_norm():
    """A chain whose state vanishes is a numeric error on this path too, and the handle stays usable."""
    import paper_2512_20064_gb300 as F

    b, ts, _ = gen.mps_tensors(6, 2, 4, base_seed=2, dtype=np.complex64)
    with F.Sampler(precision="fp32") as s:
        s.load_chain(ts)
        s.load_site(3, np.zeros_like(ts[3]))
        with pytest.raises(F.FastMPSError) as e:
            s.sample(b, 2, 40, 1)
        assert e.value.code == -8
        s.load_site(3, ts[3])
        assert np.isfinite(s.sample(b, 2, 40, 1)[1]).all()


@pytest.mark.parametrize("M,d,chi,one", [(10, 3, 16, True), (10, 2, 40, True), (13, 3, 350, False)])
def test_micro_batches_of_fp32_calls(M, d, chi, one):
    """max_microbatch bounds the rows of a launch, so a narrow chain runs in one launch only where all rows fit it (rows
    of d * 2 chi > 2048 columns never do).  Bit for bit the same for one launch, one micro-batch per site (one stream)
    and several (two streams)."""
    import paper_2512_20064_gb300 as F

    N = 1000
    b, ts, _ = gen.mps_tensors(M, d, chi, base_seed=44, skew=1.5, dtype=np.complex64)
    out = {}
    for mb in (0, 256, 1024):
        with F.Sampler(precision="fp32", max_microbatch=mb) as s:
            s.load_chain(ts)
            out[mb] = s.sample(b, d, N, 7, trace_rows=N)
            st = s.stats()
            if mb == 256:
                assert st["contract_launches"] == 4 * M
            else:
                assert st["contract_launches"] == (1 if one else M)
    for mb in (256, 1024):
        assert all(np.array_equal(x, y) for x, y in zip(out[0], out[mb])), mb


@pytest.mark.parametrize("d,chi,N,one", [
    (10, 33, 10000, False),  # ten tiles, not seven: 3.29 ms in one launch, 2.20 in two a site
    (10, 33, 131072, False),
    (2, 64, 131072, False),
    (3, 16, 10000, True),
    (2, 32, 64, True),
])
def test_narrow_chains_take_the_shorter_route(d, chi, N, one):
    import paper_2512_20064_gb300 as F

    b, ts, _ = gen.mps_tensors(24, d, chi, base_seed=8, skew=1.5, dtype=np.complex64)
    with F.Sampler(precision="fp32") as s:
        s.load_chain(ts)
        s.sample(b, d, N, 1)
        assert (s.stats()["contract_launches"] == 1) == one
