"""The default kernels of large batches at the edges of their modulus ranges,
chosen explicitly so that small inputs reach them: the largest primes below
2^30, 2^31 and 2^62 (and the smallest from 2^59), with the inputs that have the
largest sums, against the oracle."""
import numpy as np
import pytest

from oracle import native
from paper_2307_06554_gb300 import workloads as wl

from helpers import run_plan_batch

pytestmark = pytest.mark.gpu


def _primes(n, bits, low=False):
    """The largest prime q = 1 mod 2n below 2^bits, or the smallest from there."""
    step = 2 * n
    j = ((1 << bits) - 2) // step + (1 if low else 0)
    while not wl.is_prime(1 + step * j):
        j += 1 if low else -1
    return [1 + step * j]


@pytest.mark.parametrize("n,bits,low", [
    (512, 30, False), (1024, 30, False), (2048, 30, False), (4096, 30, False), (8192, 30, False), (16384, 30, False),
    (512, 31, False), (1024, 31, False), (2048, 31, False), (4096, 31, False), (8192, 31, False), (16384, 31, False),
    (32768, 31, False), (65536, 31, False), (32768, 30, False), (65536, 30, False),
    (4096, 62, False), (8192, 62, False), (16384, 62, False), (32768, 62, False), (65536, 62, False),
    (8192, 59, True), (16384, 59, True), (32768, 59, True), (65536, 59, True),
])
def test_edges(n, bits, low):
    from paper_2307_06554_gb300 import polymul as pm
    qs = _primes(n, bits, low)
    q = qs[0]
    dt = np.uint32 if bits <= 31 else np.uint64
    rng = np.random.default_rng(n + bits)
    a = wl.uniform_coeffs(rng, 4, qs, n, dt)
    b = wl.uniform_coeffs(rng, 4, qs, n, dt)
    a[0] = b[0] = q - 1
    a[1, 0, ::2], a[1, 0, 1::2], b[1] = q - 1, 0, q // 2
    got = {}
    for flags in (0, pm.FLAG_OVERLAP):
        with pm.Plan(n, qs, path=pm.PATH_NTT, flags=flags) as plan:
            got[flags, "by size"] = run_plan_batch(plan, a, b)
            plan.select(0)
            got[flags, "default"] = run_plan_batch(plan, a, b)
    js = [0, 1, n // 2, n - 2, n - 1] + [int(x) for x in rng.integers(0, n, 11)]
    for key, c in got.items():
        assert np.array_equal(c, got[0, "default"]), key
        for i in range(len(a)):
            want = native.coeffs(a[i, 0], b[i, 0], q, js)
            assert np.array_equal(c[i, 0][js].astype(np.uint64), np.asarray(want, dtype=np.uint64)), (key, i)
