"""Loading of 16-bit site tensors (needs a GB300): the device repack against the FP64 oracle at odd widths, from host
and device memory of both types, Vidal form, reloads over other shapes, and against the host conversion of the
streamed residency, which writes its 16-bit planes on the CPU."""
import numpy as np
import pytest

import gen
import parity
from oracle import quant

pytestmark = pytest.mark.gpu

BONDS = [1, 3, 7, 8, 20, 33, 64, 65, 63, 32, 11, 4, 2, 1]  # below, at and above the tiles of 32 columns and 64 rows


def _chain(dtype):
    return gen.mps_tensors(len(BONDS) - 1, 3, 65, base_seed=70, skew=1.5, dtype=dtype, bonds=BONDS)[:2]


def _stored(ts, precision):
    planes = 2 if precision in ("bf16x3", "fp16x3") else 1
    return [(quant.dequant_fp16 if precision.startswith("fp16") else quant.dequant_bf16)(A, planes) for A in ts]


@pytest.mark.parametrize("precision", ["bf16x2", "bf16x3", "fp16x2", "fp16x3"])
@pytest.mark.parametrize("dtype", [np.complex64, np.complex128])
def test_repack_sources_agree_and_match_oracle(precision, dtype):
    import torch

    import paper_2512_20064_gb300 as F

    b, ts = _chain(dtype)
    N, out = 200, {}
    for where in ("host", "device", "misaligned", "streamed"):
        with F.Sampler(precision=precision, residency="host_stream" if where == "streamed" else "hbm") as s:
            for k, A in enumerate(ts):
                if where == "host" or where == "streamed":
                    s.load_site(k, A)
                elif where == "device":
                    s.load_site(k, torch.from_numpy(A).cuda())
                else:  # a device pointer aligned to a real number only: staged, not read in place
                    flat = torch.zeros(2 * A.size + 1, dtype=torch.float32 if dtype == np.complex64 else torch.float64,
                                       device="cuda")
                    flat[1:] = torch.from_numpy(A.reshape(-1).view(A.real.dtype)).cuda()
                    torch.cuda.synchronize()
                    rc = F.load_library().fastmps_load_site(s.h, k, *A.shape, flat.data_ptr() + flat.element_size(),
                                                            F.C64 if dtype == np.complex64 else F.C128)
                    assert rc == 0
            out[where] = s.sample(b, 3, N, 9, trace_rows=N)
    for where in ("device", "misaligned", "streamed"):
        assert all(np.array_equal(x, y) for x, y in zip(out["host"], out[where])), where
    smp, lp, tr = out["host"]
    parity.check(b, _stored(ts, precision), 9, np.arange(N), smp, lp, 1e-4, dev_trace=tr, trace_rows=N)


@pytest.mark.parametrize("precision", ["fp32", "bf16x3", "fp16x2"])
def test_reload_over_other_shapes(precision):
    """Sites loaded over smaller, larger and equal ones give the results of a fresh handle; a refused load keeps
    the site that was there."""
    import paper_2512_20064_gb300 as F

    b, ts = _chain(np.complex64)
    other, to, _ = gen.mps_tensors(13, 3, 40, base_seed=90, skew=1.5, dtype=np.complex64)
    again, ta = _chain(np.complex64)
    ta = [np.ascontiguousarray(A[:, ::-1, :]) for A in ta]
    with F.Sampler(precision=precision) as s:
        for bb, tt in ((b, ts), (other, to), (b, ts), (again, ta)):
            s.load_chain(tt)
            with pytest.raises(F.FastMPSError):
                s.load_site(5, np.zeros((50, 3, 4), np.complex64))  # not an isometry shape
            got = s.sample(bb, 3, 150, 3)
            with F.Sampler(precision=precision) as fresh:
                fresh.load_chain(tt)
                want = fresh.sample(bb, 3, 150, 3)
            assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


@pytest.mark.parametrize("precision", ["bf16x3", "fp16x2"])
def test_reload_that_fails_late_keeps_the_old_site(precision, monkeypatch):
    """A load that fails after its operands were chosen (here: their tensor maps) leaves the loaded values alone,
    although a reload may take over the operands of the site that it replaces."""
    import paper_2512_20064_gb300 as F

    b, ts = _chain(np.complex64)
    with F.Sampler(precision=precision) as s:
        s.load_chain(ts)
        want = s.sample(b, 3, 150, 3)
        for k in (4, 6):
            monkeypatch.setenv("FASTMPS_TEST_FAIL_TENSOR_MAPS", "1")
            with pytest.raises(F.FastMPSError):
                s.load_site(k, np.ascontiguousarray(ts[k][:, ::-1, :]))
            monkeypatch.delenv("FASTMPS_TEST_FAIL_TENSOR_MAPS")
            got = s.sample(b, 3, 150, 3)
            assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


def test_tune_cache_of_other_kernels_is_not_read(tmp_path):
    """A choice file without the present version is measured anew (its width of 96 is no candidate); one with it is
    read and stays as it is."""
    import json
    import os
    import subprocess
    import sys

    cache = tmp_path / "tune.json"
    cache.write_text(json.dumps({"1:40:3:40": 96}))
    code = ("import sys; sys.path.insert(0, %r)\n"
            "import numpy as np, gen, paper_2512_20064_gb300 as F\n"
            "b, ts, _ = gen.mps_tensors(9, 3, 40, base_seed=4, skew=1.5, dtype=np.complex64)\n"
            "with F.Sampler(precision='bf16x2', autotune=True) as s:\n"
            "    s.load_chain(ts)\n"
            "    assert np.isfinite(s.sample(b, 3, 300, 1)[1]).all()\n") % os.path.dirname(os.path.dirname(__file__))
    texts = []
    for _ in range(2):
        subprocess.run([sys.executable, "-c", code], env=dict(os.environ, FASTMPS_TUNE_CACHE=str(cache)), check=True,
                       timeout=300)
        texts.append(cache.read_text())
    table = json.loads(texts[0])
    assert table["1:40:3:40"] == 64 and "version" in table  # 64 columns: the only candidate not wider than the block
    assert texts[0] == texts[1]
