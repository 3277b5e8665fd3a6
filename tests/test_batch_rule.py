"""Plans that run another kernel for some batch sizes: batches on every side of
the lines, in turn on one stream (launches of different kernels share the
plan's work counter), with and without POLYMUL_FLAG_OVERLAP, against the
default kernel chosen explicitly, which in turn is checked against the oracle.
`lines` are in products per SM; the one product more or less falls on either
side."""
import numpy as np
import pytest

from oracle import native
from paper_2307_06554_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# n, q or bits, lines (products per SM) of overlapped and of other plans
CASES = [
    (256, 3329, (3500 / 256,)),          # auxiliary prime
    (256, 7681, (4500 / 256, 4800 / 256, 32, 39)),  # smallest moduli
    (512, 12289, (4500 / 512, 4800 / 512)),
    (1024, 12289, (4500 / 1024, 4600 / 1024)),
    (512, 30, (4,)),
    (1024, 30, (2,)),
    (1024, 31, (2,)),
    (2048, 30, (1,)),
    (2048, 31, (1,)),
    (4096, 17, (3, 9)),
    (4096, 31, (9,)),
    (4096, 30, (9,)),
    (8192, 31, (1, 15 / 8, 2, 13 / 4)),
    (8192, 30, (1, 15 / 8, 2, 13 / 4)),
    (8192, 17, (1, 2)),
    (16384, 31, (1 / 2,)),
    (8192, 59, (1 / 2,)),
    (16384, 61, (1 / 4,)),
]


@pytest.mark.parametrize("overlap", [False, True])
@pytest.mark.parametrize("n,q,lines", CASES)
def test_both_sides(n, q, lines, overlap):
    import torch
    from paper_2307_06554_gb300 import polymul as pm
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if q > 64:
        qs, dt = [q], torch.int32
    else:
        qs = wl.draw_primes(np.random.default_rng(n + q), 1, q, q, n.bit_length())
        dt = torch.int32 if q <= 31 else torch.int64
    sizes = [1]
    for x in lines:
        at = int(x * sms)
        sizes += [at + 1, at, 2]
    most = max(sizes)
    gen = torch.Generator(device="cuda").manual_seed(n)
    a, b = (torch.randint(0, 1 << 62, (most, 1, n), generator=gen, device="cuda").remainder_(qs[0]).to(dt)
            for _ in range(2))
    a[0] = b[0] = qs[0] - 1
    with pm.Plan(n, qs, path=pm.PATH_NTT) as plan:
        plan.select(0)
        want = torch.empty_like(a)
        plan.batch(a, b, want)
        torch.cuda.synchronize()
    pick = [0, most // 2, most - 1]
    npt = np.uint32 if dt == torch.int32 else np.uint64
    host = [x[pick].cpu().numpy().view(npt) for x in (a, b, want)]
    assert np.array_equal(host[2].astype(np.uint64), native.polymul_batch(host[0], host[1], qs))
    st = torch.cuda.Stream()
    outs = [torch.full((s, 1, n), -1, dtype=dt, device="cuda") for s in sizes]
    with pm.Plan(n, qs, path=pm.PATH_NTT, flags=pm.FLAG_OVERLAP if overlap else 0) as plan:
        torch.cuda.synchronize()
        for _ in range(3):
            for s, c in zip(sizes, outs):
                plan.batch(a[:s], b[:s], c, stream=st.cuda_stream)
        pm.polymul_plan_status(plan.handle, st.cuda_stream)
        torch.cuda.synchronize()
    for s, c in zip(sizes, outs):
        assert torch.equal(c, want[:s]), s
