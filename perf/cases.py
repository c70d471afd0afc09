"""The work that users of this library have it do, as measurable cases.

Every case is one call (or one load followed by a call) through the Python binding of
``paper_2512_20064_gb300``.  Site tensors are seeded Haar-random isometries with the physical index
skewed by exp(-s / 1.5), the bond profile is min(d^k, d^(M-k), chi), and the interior sites share a
pool of two tensors (a chain may reuse its tensors; the path does the same work for each site).

Kinds
  sample        draw N rows of a resident chain (every precision, host or device outputs)
  displaced     the same with per-sample displacement amplitudes (host or device amplitudes)
  streamed      site tensors in pinned host memory, copied per site while the previous one computes
  batch         several independent chains in one call
  load          load a chain of new site tensors from device memory, then draw a few rows of it
  displacement  displacement matrices of N amplitudes
"""
import math

import numpy as np
import torch

import paper_2512_20064_gb300 as F

SKEW = 1.5
POOL = 2


def listed():
    return [
        # one request of a sampling service: few rows of a short chain, default options, host outputs
        dict(name="request_fp32", kind="sample", precision="fp32", chunk=0, M=64, d=2, chi=32, N=64, out="host"),
        # the smallest full workload: 10^4 rows of a 12-site chain
        dict(name="tiny_fp32", kind="sample", precision="fp32", chunk=0, M=12, d=3, chi=16, N=10000, out="host"),
        # the plain workload on complex64 tensors (fewer sites and rows)
        dict(name="plain_fp32", kind="sample", precision="fp32", chunk=0, M=48, d=4, chi=256, N=1 << 15, out="device"),
        # the plain workload on the tensor cores, at its full row count
        dict(name="plain_bf16x2", kind="sample", precision="bf16x2", chunk=0, M=128, d=4, chi=256, N=1 << 17,
             out="device"),
        # the precision workload's shape and mode: 16-bit tensors, promoted accumulation
        dict(name="precision_fp16x2", kind="sample", precision="fp16x2", chunk=4, M=40, d=4, chi=1024, N=1 << 16,
             out="device"),
        # a chain of odd width within the accuracy bound of the original tensors, odd row count, host outputs
        dict(name="ragged_fp16x3", kind="sample", precision="fp16x3", chunk=4, M=33, d=3, chi=777, N=5003,
             out="host"),
        # lossy Gaussian boson sampling: a displacement per sample and site, amplitudes resident
        dict(name="gbs_bf16x2", kind="displaced", precision="bf16x2", M=64, d=4, chi=256, N=1 << 16, mu="device",
             sigma=0.3, out="device"),
        # the same on complex64 tensors: more photons, an odd width, few rows, amplitudes on the host
        dict(name="gbs_ragged_fp32", kind="displaced", precision="fp32", M=32, d=6, chi=90, N=3001, mu="host",
             sigma=0.6, out="host"),
        # a wide chain whose tensors are streamed from the host (the knee study's width)
        dict(name="streamed_bf16x2", kind="streamed", precision="bf16x2", chunk=0, M=24, d=3, chi=2000, N=1 << 13,
             out="host"),
        # independent chains of different shapes in one call
        dict(name="batch_bf16x2", kind="batch", precision="bf16x2", jobs=10, recipe=2025, out="device"),
        # a new chain arrives in Vidal form: load it, draw a few rows
        dict(name="load_vidal_fp16x2", kind="load", precision="fp16x2", chunk=4, vidal=True, M=20, d=4, chi=512,
             N=256, out="host"),
        # displacement matrices of four million amplitudes
        dict(name="displacement_d4", kind="displacement", d=4, N=1 << 22, sigma=0.3),
    ]


# ---------------------------------------------------------------------------------------------------
# drawn cases
# ---------------------------------------------------------------------------------------------------
# rough cost of one pass, in seconds, from the flops of a case (what the modes reach on one GPU)
_RATE = {"fp32": 4.5e13, "bf16x2": 7e14, "bf16x3": 4.5e14, "bf16x3l": 4.5e14, "fp16x2": 6.5e14, "fp16x3": 4.5e14}
_MAX_S = 0.06


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _rows(rng, c, lo, hi):
    """A row count in [lo, hi], log-uniform, whose pass costs at most _MAX_S."""
    b = _bonds(c["M"], c["d"], c["chi"])
    per_row = sum(8.0 * b[k] * c["d"] * b[k + 1] for k in range(c["M"])) / _RATE[c["precision"]]
    hi = max(lo + 1, min(hi, int(_MAX_S / per_row)))
    return _log(rng, lo, hi)


def draw(rng):
    kind = rng.choice(["sample", "sample", "sample", "displaced", "streamed", "batch", "load", "displacement"])
    out = rng.choice(["host", "device"])
    if kind == "sample":
        precision, chunk = rng.choice([("fp32", 0), ("fp32", 0), ("bf16x2", 0), ("bf16x2", 0), ("bf16x3", 0),
                                       ("bf16x3l", 0), ("fp16x2", 4), ("fp16x2", 4), ("fp16x2", 0), ("fp16x3", 4)])
        c = dict(kind=kind, precision=precision, chunk=chunk, M=_log(rng, 8, 128), d=rng.choice([2, 3, 4, 6, 10]),
                 chi=_log(rng, 8, 1200), out=out)
        c["N"] = _rows(rng, c, 1, 1 << 17)
    elif kind == "displaced":
        c = dict(kind=kind, precision=rng.choice(["fp32", "bf16x2"]), M=_log(rng, 8, 64), d=rng.choice([2, 3, 4, 6, 10]),
                 chi=_log(rng, 16, 400), mu=rng.choice(["host", "device"]), sigma=round(rng.uniform(0.2, 0.6), 3),
                 out=out)
        c["N"] = _rows(rng, c, 16, 1 << 16)
    elif kind == "streamed":
        c = dict(kind=kind, precision=rng.choice(["bf16x2", "bf16x3", "fp16x2"]), chunk=0, M=_log(rng, 8, 24),
                 d=rng.choice([2, 3, 4]), chi=_log(rng, 200, 1600), out=out)
        c["N"] = _rows(rng, c, 128, 1 << 14)
    elif kind == "batch":
        c = dict(kind=kind, precision=rng.choice(["bf16x2", "bf16x3"]), jobs=rng.randint(3, 10),
                 recipe=rng.randrange(1 << 20), out=out)
    elif kind == "load":
        c = dict(kind=kind, precision=rng.choice(["fp32", "bf16x2", "fp16x2", "fp16x3"]), chunk=0,
                 vidal=rng.random() < 0.5, M=_log(rng, 8, 32), d=rng.choice([2, 3, 4, 6]), chi=_log(rng, 30, 700),
                 out=out)
        c["N"] = _log(rng, 16, 512)
    else:
        c = dict(kind=kind, d=rng.choice([3, 4, 5, 6, 8, 10]), sigma=round(rng.uniform(0.2, 0.6), 3))
        c["N"] = _log(rng, 1 << 10, (1 << 26) // (c["d"] * c["d"]))
    return c


# ---------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------
def _bonds(M, d, chi):
    left, right = [1], [1]
    for _ in range(M):
        left.append(min(left[-1] * d, chi))
        right.append(min(right[-1] * d, chi))
    return [min(left[k], right[M - k]) for k in range(M + 1)]


def _isometry(seed, cl, d, cr):
    g = torch.Generator(device="cuda").manual_seed(seed)
    z = torch.randn((d * cr, cl, 2), generator=g, device="cuda", dtype=torch.float32)
    z = z * torch.exp(-torch.arange(d, device="cuda") / SKEW).repeat_interleave(cr)[:, None, None]
    q, r = torch.linalg.qr(torch.view_as_complex(z))
    ph = torch.diagonal(r)
    q = q * (ph / ph.abs())[None, :]
    return q.transpose(0, 1).reshape(cl, d, cr).contiguous()


def _chain(M, d, chi, seed):
    """(bonds, tensors, index): the interior sites share POOL tensors, the others have their own."""
    b = _bonds(M, d, chi)
    tensors, index, pool = [], [], {}
    for k in range(M):
        j = k % POOL if b[k] == chi and b[k + 1] == chi else None
        if j is not None and j in pool:
            index.append(pool[j])
            continue
        if j is not None:
            pool[j] = len(tensors)
        index.append(len(tensors))
        tensors.append(_isometry(seed * 4099 + k, b[k], d, b[k + 1]))
    return b, tensors, index


def _jobs(case):
    """Shapes of the chains of a batch: M, d, chi and N of each, spread as in the batching workload."""
    r = np.random.Generator(np.random.PCG64(case["recipe"]))
    jobs = []
    for _ in range(case["jobs"]):
        jobs.append(dict(M=int(r.integers(12, 72)), d=int(r.choice([2, 3, 4, 6])),
                         chi=int(round(math.exp(r.uniform(math.log(32), math.log(400))))),
                         N=int(round(math.exp(r.uniform(math.log(200), math.log(8000)))))))
    return jobs


def _amplitudes(case, seed, shape):
    g = torch.Generator(device="cuda").manual_seed(seed * 31 + 17)
    z = torch.randn((*shape, 2), generator=g, device="cuda", dtype=torch.float32)
    return torch.view_as_complex(z * (case["sigma"] / math.sqrt(2.0)))


def _vidal(tensors, seed):
    """Gamma_k = A_k / Lambda_k with decaying normalised spectra Lambda_k (real, of the bond right of site k)."""
    gammas, lams = [], []
    for A in tensors:
        cr = A.shape[2]
        lam = torch.exp(-3.0 * torch.arange(cr, device="cuda", dtype=torch.float32) / cr)
        lam = lam / lam.norm()
        gammas.append((A / lam).contiguous())
        lams.append(lam)
    return gammas, lams


def _outputs(case, N, M):
    if case["out"] == "device":
        return dict(out_samples=torch.empty((N, M), dtype=torch.uint8, device="cuda"),
                    out_logprob=torch.empty(N, dtype=torch.float64, device="cuda"))
    return {}


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=1000 + seed % 100003)
    if kind == "displacement":
        st["mu"] = _amplitudes(case, seed, (case["N"],))
        st["D"] = torch.empty((case["d"], case["d"], case["N"]), dtype=torch.complex64, device="cuda")
        torch.cuda.synchronize()
        st["sampler"] = F.Sampler()
        return st
    if kind == "batch":
        st["runner"] = F.Sampler(precision=case["precision"])
        st["samplers"], st["jobs"] = [], []
        for j, p in enumerate(_jobs(case)):
            b, ts, idx = _chain(p["M"], p["d"], p["chi"], seed * 64 + j)
            torch.cuda.synchronize()
            s = F.Sampler(precision=case["precision"])
            s.load_chain(ts, idx)
            o = _outputs(case, p["N"], p["M"])
            if not o:
                o = dict(out_samples=np.empty((p["N"], p["M"]), np.uint8), out_logprob=np.empty(p["N"], np.float64))
            st["samplers"].append(s)
            st["jobs"].append(dict(chain=s.h, bonds=b, d=p["d"], N=p["N"], seed=st["seed"] + j, job=j, **o))
        return st
    b, ts, idx = _chain(case["M"], case["d"], case["chi"], seed)
    torch.cuda.synchronize()
    st["bonds"] = b
    st["sampler"] = F.Sampler(precision=case["precision"], accum_chunk=case.get("chunk", 0),
                              residency="host_stream" if kind == "streamed" else "hbm")
    st["out"] = _outputs(case, case["N"], case["M"])
    if kind == "load":
        ts = [ts[j] for j in idx]
        if case["vidal"]:
            st["gammas"], st["lams"] = _vidal(ts, seed)
        else:
            st["tensors"] = ts
        torch.cuda.synchronize()
        return st
    st["sampler"].load_chain(ts, idx)
    if kind == "displaced":
        mu = _amplitudes(case, seed, (case["M"], case["N"]))
        st["mu"] = mu if case["mu"] == "device" else mu.cpu().numpy()
    return st


# ---------------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "displacement":
        return F.fastmps_displacement(state["sampler"].h, state["mu"], case["d"], out=state["D"])
    if kind == "batch":
        F.fastmps_sample_batch(state["runner"].h, state["jobs"])
        return [(j["out_samples"], j["out_logprob"]) for j in state["jobs"]]
    s = state["sampler"]
    if kind == "load":
        if case["vidal"]:
            s.load_chain_vidal(state["gammas"], state["lams"])
        else:
            s.load_chain(state["tensors"])
    return s.sample(state["bonds"], case["d"], case["N"], state["seed"], mu=state.get("mu"), **state["out"])


# ---------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------------
def _flops(b, d, N):
    return sum(8.0 * b[k] * d * b[k + 1] for k in range(len(b) - 1)) * N


def _stored(precision):
    """Bytes of one stored complex entry of a site tensor."""
    return 8 if precision == "fp32" else 8 if precision in ("bf16x3", "bf16x4", "fp16x3") else 4


def _tensor_entries(b, d, chi):
    n, pool = 0, set()
    for k in range(len(b) - 1):
        if b[k] == chi and b[k + 1] == chi:
            if k % POOL in pool:
                continue
            pool.add(k % POOL)
        n += b[k] * d * b[k + 1]
    return n


def work(case):
    if case["kind"] == "displacement":
        d = case["d"]
        return dict(bytes=8.0 * case["N"] * (1 + d * d), flops=8.0 * case["N"] * d * d)
    if case["kind"] == "batch":
        w = [work(dict(kind="sample", precision=case["precision"], **p)) for p in _jobs(case)]
        return dict(bytes=sum(x["bytes"] for x in w), flops=sum(x["flops"] for x in w))
    M, d, N = case["M"], case["d"], case["N"]
    b = _bonds(M, d, case["chi"])
    if case["kind"] == "load":  # each site's tensor is an input of its own, read as complex64, stored once, read once
        n = sum(b[k] * d * b[k + 1] for k in range(M))
        return dict(bytes=n * (8.0 + 2 * _stored(case["precision"])) + N * (M + 8), flops=_flops(b, d, N))
    n = _tensor_entries(b, d, case["chi"])
    more = 8.0 * M * N if case["kind"] == "displaced" else 0.0
    return dict(bytes=n * _stored(case["precision"]) + N * (M + 8.0) + more, flops=_flops(b, d, N))


# ---------------------------------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------------------------------
def _uniforms(seed, N, k, job):
    """Philox4x32-10 with key (seed lo, seed hi) and counter (n lo, n hi, k, job); 53 bits of the first two words."""
    m32 = np.uint64(0xFFFFFFFF)
    n = np.arange(N, dtype=np.uint64)
    c = [n & m32, n >> np.uint64(32), np.full(N, k, np.uint64), np.full(N, job, np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        a, z = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(z >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), z & m32, (a >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), a & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    bits = (c[0] << np.uint64(21)) | (c[1] >> np.uint64(11))
    return torch.from_numpy((bits.astype(np.float64) + 0.5) * 2.0**-53).cuda()


def _as_stored(A, precision):
    """The values that the store of a precision holds, in complex128."""
    if precision == "fp32":
        return A.to(torch.complex128)
    x = torch.view_as_real(A.to(torch.complex64)).contiguous()
    kind, scale = torch.bfloat16, 1.0
    if precision.startswith("fp16"):
        kind, scale = torch.float16, 2.0 ** math.floor(math.log2(32768.0 / float(x.abs().max())))
        x = x * scale
    hi = x.to(kind)
    v = hi.double()
    if precision in ("bf16x3", "bf16x4", "fp16x3"):
        v = v + (x - hi.float()).to(kind).double()
    return torch.view_as_complex(v / scale)


def _matrices(mu, d):
    """exp(-|mu|^2/2) exp(mu a^+) exp(-mu^* a) of every amplitude, shape (d, d) + mu.shape."""
    mu = mu.to(torch.complex128)
    f = [math.factorial(i) for i in range(d)]
    pw, pc = [torch.ones_like(mu)], [torch.ones_like(mu)]
    for _ in range(d - 1):
        pw.append(pw[-1] * mu)
        pc.append(pc[-1] * -mu.conj())
    g = torch.exp(-0.5 * mu.abs() ** 2)
    D = torch.empty((d, d, *mu.shape), dtype=torch.complex128, device=mu.device)
    for s in range(d):
        for t in range(d):
            z = torch.zeros_like(mu)
            for m in range(min(s, t) + 1):
                z += (math.sqrt(f[s] / f[m]) / math.factorial(s - m) * math.sqrt(f[t] / f[m]) / math.factorial(t - m)
                      ) * pw[s - m] * pc[t - m]
            D[s, t] = g * z
    return D


def _sample64(b, tensors, index, d, N, seed, job=0, mu=None):
    M = len(b) - 1
    v = torch.ones((N, 1), dtype=torch.complex128, device="cuda")
    logp = torch.zeros(N, dtype=torch.float64, device="cuda")
    out = torch.empty((N, M), dtype=torch.uint8, device="cuda")
    rows = torch.arange(N, device="cuda")
    for k in range(M):
        A = tensors[index[k]]
        y = (v @ A.reshape(b[k], d * b[k + 1])).reshape(N, d, b[k + 1])
        if mu is not None:
            y = torch.einsum("stn,ntb->nsb", _matrices(mu[k], d), y)
        w = torch.view_as_real(y).square().sum((2, 3))
        C = w.cumsum(1)
        u = _uniforms(seed, N, k, job)
        s = (C[:, :-1] < (u * C[:, -1])[:, None]).sum(1)
        ws = w[rows, s]
        logp += torch.log(ws / C[:, -1])
        v = y[rows, s] / ws.sqrt()[:, None]
        out[:, k] = s.to(torch.uint8)
    return out, logp


def exact(case, seed):
    if case["kind"] == "displacement":
        mu = _amplitudes(case, seed, (case["N"],))
        return _matrices(mu, case["d"])
    if work(case)["flops"] > 4e12:
        return None
    s0 = 1000 + seed % 100003
    if case["kind"] == "batch":
        got = []
        for j, p in enumerate(_jobs(case)):
            b, ts, idx = _chain(p["M"], p["d"], p["chi"], seed * 64 + j)
            _, lp = _sample64(b, [_as_stored(A, case["precision"]) for A in ts], idx, p["d"], p["N"], s0 + j, job=j)
            got.append((None, lp))
        return got
    b, ts, idx = _chain(case["M"], case["d"], case["chi"], seed)
    if case["kind"] == "load" and case["vidal"]:
        gammas, lams = _vidal(ts, seed)
        ts = [(G * L).to(torch.complex64) for G, L in zip(gammas, lams)]
    mu = _amplitudes(case, seed, (case["M"], case["N"])) if case["kind"] == "displaced" else None
    _, lp = _sample64(b, [_as_stored(A, case["precision"]) for A in ts], idx, case["d"], case["N"], s0, mu=mu)
    return None, lp
