"""The shape set that an uneven list takes by its sizes: lists on both sides of
each line, pools below 2^30 (Harvey bounds) and with 31-bit primes, sampled
against the oracle and equal under the other set.  Set 0 runs one CTA per SM,
set 1 two."""
import numpy as np
import pytest

from oracle import native
from paper_2307_06554_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# (degrees, coefficients per SM, set)
LISTS = [
    ((1024,), 1000, 0),
    ((8192,), 17000, 0),
    ((8192,), 21000, 1),
    ((1024, 8192), 17000, 0),   # half of the coefficients at 2^13
    ((1024, 8192), 21000, 1),
    ((1024, 2048, 4096), 36000, 0),
    ((1024, 2048, 4096), 44000, 1),
    ((2048, 4096), 44000, 0),
    ((2048, 4096), 104000, 1),
]


@pytest.mark.parametrize("bits", [30, 31])
@pytest.mark.parametrize("degrees,per_sm,which", LISTS)
def test_set_by_size(degrees, per_sm, which, bits):
    import torch
    from paper_2307_06554_gb300 import polymul as pm
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(per_sm + bits)
    pool = wl.draw_primes(rng, 5, bits, bits, 14)
    products = []
    share = per_sm * sms // len(degrees)
    for n in degrees:
        rows = share // n
        while rows:
            k = min(rows, 5)
            products.append((n, np.sort(rng.permutation(5)[:k]).astype(np.uint32)))
            rows -= k
    q = np.array(pool, dtype=np.int64)
    rows_q = np.concatenate([np.repeat(q[idx.astype(np.int64)], n) for n, idx in products])
    rows_q = torch.from_numpy(rows_q).cuda()
    gen = torch.Generator(device="cuda").manual_seed(per_sm)
    ta, tb = ((torch.randint(0, 1 << 62, rows_q.shape, generator=gen, device="cuda") % rows_q).to(torch.int32)
              for _ in range(2))
    with pm.Ragged(pool, 8192, products) as r:
        units, grid = r.info["units"], r.info["grid"]
        cap = (2 if which else 1) * sms
        assert grid == min(cap, units)
        tc = torch.full_like(ta, -1)
        r.run(ta, tb, tc)
        pm.polymul_ragged_status(r.batch)
        r.select(1 - which)
        other = torch.full_like(ta, -1)
        r.run(ta, tb, other)
        pm.polymul_ragged_status(r.batch)
        assert torch.equal(tc, other)
        offsets = list(r.offsets)
    a, b, c = (x.cpu().numpy().view(np.uint32) for x in (ta, tb, tc))
    for i in sorted({0, len(products) // 2, len(products) - 1}):
        n, idx = products[i]
        s = slice(offsets[i], offsets[i] + n * len(idx))
        want = native.polymul_batch(a[s].reshape(1, len(idx), n), b[s].reshape(1, len(idx), n), [pool[j] for j in idx])
        assert np.array_equal(c[s].reshape(len(idx), n), want[0].astype(np.uint32)), i
