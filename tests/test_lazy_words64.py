"""64-bit words with moduli below 2^59 (values up to 32q between reductions),
at the edges: the largest primes below the limit, inputs with the largest
sums, every degree's default kernel and its few-products form, against the
CPU oracle up to n = 2^13 and against the Harvey-bound candidate above."""
import numpy as np
import pytest

from oracle import native
from paper_2307_06554_gb300 import workloads as wl

from helpers import assert_equal_residues, run_plan_batch

pytestmark = pytest.mark.gpu


def _top_primes(n, count=2):
    """The largest primes q = 1 mod 2n below 2^59."""
    out, j = [], ((1 << 59) - 2) // (2 * n)
    while len(out) < count:
        if wl.is_prime(1 + 2 * n * j):
            out.append(1 + 2 * n * j)
        j -= 1
    return out


def _extremes(rng, batch, qs, n):
    a = wl.uniform_coeffs(rng, batch, qs, n, np.uint64)
    b = wl.uniform_coeffs(rng, batch, qs, n, np.uint64)
    for j, q in enumerate(qs):
        a[0, j] = b[0, j] = q - 1
        a[1, j, ::2] = q - 1
        a[1, j, 1::2] = 0
        b[1, j] = q // 2
    return a, b


@pytest.mark.parametrize("logn", range(4, 14))
def test_against_oracle(logn):
    from paper_2307_06554_gb300 import polymul as pm
    n = 1 << logn
    qs = _top_primes(n)
    rng = np.random.default_rng(logn)
    a, b = _extremes(rng, 3, qs, n)
    want = native.polymul_batch(a, b, qs)
    with pm.Plan(n, qs, path=pm.PATH_NTT) as plan:
        assert plan.info["ntt_mode"] == 4
        for c in range(plan.info["candidates"]):
            assert_equal_residues(run_plan_batch(plan, a, b), want, "n=%d before candidate %d" % (n, c))
            plan.select(c)
        assert_equal_residues(run_plan_batch(plan, a, b), want, "n=%d last candidate" % n)


@pytest.mark.parametrize("n,batch", [(16384, 4), (16384, 41), (32768, 4), (32768, 21), (65536, 3)])
def test_large_degrees(n, batch):
    """Every candidate of the plan (the default or, for few products, its
    small form first) agrees; from 2^15 one of them is a Harvey-bound kernel."""
    from paper_2307_06554_gb300 import polymul as pm
    qs = _top_primes(n)
    rng = np.random.default_rng(n + batch)
    a, b = _extremes(rng, batch, qs, n)
    with pm.Plan(n, qs, path=pm.PATH_NTT) as plan:
        want = run_plan_batch(plan, a, b)
        modes = set()
        for c in range(plan.info["candidates"]):
            modes.add(plan.select(c)["ntt_mode"])
            assert np.array_equal(run_plan_batch(plan, a, b), want), "candidate %d" % c
        assert modes == ({4} if n == 16384 else {1, 4})
    # all-(q-1) squared in x^n + 1: coefficient i is 2 i + 2 - n mod q
    for j, q in enumerate(qs):
        i = np.arange(n, dtype=object)
        assert np.array_equal(want[0, j].astype(object), (2 * i + 2 - n) % q)
