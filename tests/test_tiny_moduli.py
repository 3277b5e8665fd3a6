"""The NTT unit of the smallest moduli (q < 18500, n = 2^8 .. 2^10: signed
residues, a transform that stops at polynomials of eight coefficients),
against the CPU oracle at the edges of its range: the smallest and the
largest modulus it takes, both rings, several primes, batches that leave
warps, CTAs and SMs without a unit, and the inputs with the largest partial
sums (every coefficient q - 1, or q // 2 beside q // 2 + 1)."""
import numpy as np
import pytest

from oracle import native
from paper_2307_06554_gb300 import workloads as wl

from helpers import assert_equal_residues, run_plan_batch

pytestmark = pytest.mark.gpu

LIMIT = 18500  # exclusive


def _primes(n):
    qs = [q for q in range(2 * n + 1, LIMIT, 2 * n) if wl.is_prime(q)]
    return sorted({qs[0], qs[len(qs) // 2], qs[-1]})


@pytest.mark.parametrize("cyclic", [False, True])
@pytest.mark.parametrize("n", [256, 512, 1024])
@pytest.mark.parametrize("batch", [4, 37, 1301])
def test_edges(n, batch, cyclic):
    from paper_2307_06554_gb300 import polymul as pm
    qs = _primes(n)
    rng = np.random.default_rng(n + batch)
    a = wl.uniform_coeffs(rng, batch, qs, n, np.uint32)
    b = wl.uniform_coeffs(rng, batch, qs, n, np.uint32)
    for j, q in enumerate(qs):
        a[0, j] = b[0, j] = q - 1
        a[1, j] = q // 2
        b[1, j] = q // 2 + 1
        a[2, j, ::2] = 0
        a[2, j, 1::2] = q - 1
        b[2, j] = a[2, j]
        a[3, j] = 0
        a[3, j, n - 1] = q - 1
    with pm.Plan(n, qs, path=pm.PATH_NTT, flags=pm.FLAG_CYCLIC if cyclic else 0) as plan:
        assert (plan.info["radix_bits"], plan.info["exchange_pad"]) == (5, 3)  # the default is this unit
        default = run_plan_batch(plan, a, b)  # the smaller batches run candidate 1
        plan.select(0)  # this unit whatever the batch
        got = run_plan_batch(plan, a, b)
    assert np.array_equal(got, default)
    idx = sorted(set(range(4)) | {batch // 2, batch - 2, batch - 1})
    assert_equal_residues(got[idx], native.polymul_batch(a[idx], b[idx], qs, cyclic=cyclic), "tiny moduli")
    with pm.Plan(n, qs, path=pm.PATH_NTT, flags=pm.FLAG_CYCLIC if cyclic else 0) as plan:
        plan.select(1)  # the radix-16 kernel in 32-bit residues
        assert np.array_equal(got, run_plan_batch(plan, a, b))


def test_first_modulus_past_the_limit():
    """Primes at and above the limit take the other kernels."""
    from paper_2307_06554_gb300 import polymul as pm
    q = next(q for q in range(512 * (LIMIT // 512 + 1) + 1, 1 << 20, 512) if wl.is_prime(q))
    with pm.Plan(256, [q], path=pm.PATH_NTT) as plan:
        assert plan.info["radix_bits"] == 4


@pytest.mark.parametrize("batch", [1, 9, 611, 2600])
@pytest.mark.parametrize("qs", [[12289], [18433, 12289]])
@pytest.mark.parametrize("cyclic", [False, True])
def test_shared_operand(batch, qs, cyclic):
    """One operand for the whole batch: fewer products than warps, a last
    group with idle warps, several products per warp, two primes."""
    import torch
    from paper_2307_06554_gb300 import polymul as pm
    n = 1024
    rng = np.random.default_rng(batch + len(qs))
    a = wl.uniform_coeffs(rng, 1, qs, n, np.uint32)
    b = wl.uniform_coeffs(rng, batch, qs, n, np.uint32)
    for j, q in enumerate(qs):
        a[0, j, ::3] = q - 1
        b[0, j] = q - 1
    flags = pm.FLAG_CYCLIC if cyclic else 0
    with pm.Plan(n, qs, path=pm.PATH_NTT, flags=flags) as plan:
        ta, tb = (torch.from_numpy(x.view(np.int32)).cuda() for x in (a[0].copy(), b))
        tc = torch.full_like(tb, -1)
        pm.polymul_batch_shared(plan.handle, ta, tb, tc, batch)
        torch.cuda.synchronize()
        pm.polymul_plan_status(plan.handle)
        got = tc.cpu().numpy().view(np.uint32)
        full = np.broadcast_to(a, b.shape).copy()
        assert np.array_equal(got, run_plan_batch(plan, full, b))
    idx = sorted({0, batch // 2, batch - 1})
    assert_equal_residues(got[idx], native.polymul_batch(full[idx], b[idx], qs, cyclic=cyclic), "shared tiny")
