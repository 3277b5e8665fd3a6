"""The bounds of the smallest moduli's multiplication (ntt_tiny_arith.h).

On the host: the multiplication itself, compiled from the library's headers,
over every root word and the factors at the end of its range.  On the GPU:
products whose transforms are chosen so that the inverse stages, which double
without reducing, reach the largest sums.  With b = 1 the products of the
small rings are a's own values, so a is the inverse transform of +-(q - 1)/2
in same-sign blocks of 1 .. n/8 rings, and the result has to be a itself."""
import subprocess

import numpy as np
import pytest

from paper_2307_06554_gb300 import workloads as wl
from paper_2307_06554_gb300.build import CSRC

from helpers import run_plan_batch

LIMIT = 18500  # exclusive

HOST = r"""
#include <cstdio>
#include <cstdlib>
#include "ntt_tiny_arith.h"
using namespace pm;
static long bad = 0;
static void check(int a, uint32_t w, uint32_t word, const TinyMod& m) {
  const int r = tiny_mul(a, (int)word, m);
  const long long d = (long long)a * w - r;
  if (d % m.q != 0 || r > (m.q - 1) / 2 || r < -((m.q - 1) / 2)) {
    if (bad++ == 0) printf("q=%d a=%d w=%u: %d\n", m.q, a, w, r);
  }
}
int main(int argc, char** argv) {
  for (int i = 1; i < argc; ++i) {
    const uint32_t q = (uint32_t)atoi(argv[i]);
    const TinyMod m{(int)q, (int)(uint32_t)host::inv_pow2_64(q)};
    const int h = (q - 1) / 2, lim = kTinyLim * h;
    uint32_t big[2] = {0, 0};  // the words of W = h and W = -h
    for (uint32_t w = 1; w < q; ++w) {
      const uint32_t word = tiny_word(w, q);
      for (int d = 0; d < 8; ++d) check(lim - d, w, word, m), check(d - lim, w, word, m);
      const int W = (int)(((uint64_t)q - (uint64_t)w * ((1ull << 32) % q) % q) % q);
      if (W == h) big[0] = w;
      if (W == (int)q - h) big[1] = w;
    }
    for (uint32_t w : big) {
      const uint32_t word = tiny_word(w, q);
      for (int a = -lim; a <= lim; ++a) check(a, w, word, m);
    }
  }
  return bad != 0;
}
"""


def _primes(step, lo=0):
    return [q for q in range(step + 1, LIMIT, step) if q >= lo and wl.is_prime(q)]


def build_host(tmp_path, flags):
    """The host program over the library's headers."""
    src, exe = tmp_path / "tiny.cpp", tmp_path / "tiny"
    src.write_text(HOST)
    subprocess.check_call(["g++", "-std=c++17", "-O2", *flags, "-I", CSRC, str(src), "-o", str(exe)])
    return str(exe)


def test_multiplication_over_its_range(tmp_path):
    qs = _primes(256)  # every modulus the unit takes (cyclic n = 256: q = 1 mod 256)
    assert 12289 in qs and 18433 in qs
    exe = build_host(tmp_path, ["-fwrapv"])
    r = subprocess.run([exe, *map(str, qs)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_no_signed_overflow(tmp_path):
    """The low product wraps in unsigned arithmetic: built with traps on signed
    overflow, the same range runs through."""
    exe = build_host(tmp_path, ["-fsanitize=signed-integer-overflow", "-fsanitize-undefined-trap-on-error"])
    r = subprocess.run([exe, "7681", "12289", "18433"], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)


def _root(q, order):
    """The library's root: the smallest base whose power has exactly this order."""
    for g in range(2, q):
        r = pow(g, (q - 1) // order, q)
        if pow(r, order // 2, q) == q - 1:
            return r


def _bitrev(x, bits):
    return int(format(x, "0%db" % bits)[::-1], 2) if bits else 0


def _inverse(vals, q, n, cyclic):
    """Polynomials (rows) whose residues modulo the n/8 rings x^8 - z, in the
    order of the unit's tree, are vals (rows, n/8, 8)."""
    m = n // 8
    logm = m.bit_length() - 1
    psi = _root(q, m if cyclic else 2 * m)
    x = vals.astype(np.int64) % q
    level = m // 2  # nodes of the level above
    while level:
        x = x.reshape(len(vals), level, 2, -1)
        out = np.empty((len(vals), level, 2, x.shape[-1]), dtype=np.int64)
        for g in range(level):
            i = level + g
            e = _bitrev(g, logm) // 2 if cyclic else _bitrev(i, logm)
            w = pow(psi, e, q)  # the children are modulo y - w and y + w
            lo, hi = x[:, g, 0], x[:, g, 1]
            half = pow(2, -1, q)
            out[:, g, 0] = (lo + hi) * half % q
            out[:, g, 1] = (lo - hi) % q * half % q * pow(w, -1, q) % q
        x = out
        level //= 2
    return x.reshape(len(vals), n)


def _patterns(q, n, rng):
    """Ring values of size (q - 1)/2 with the signs that let sums grow."""
    m, h = n // 8, (q - 1) // 2
    rows = []
    block = 1
    while block <= m:
        sign = np.where(np.arange(m) // block % 2 == 0, 1, -1)
        for s in (sign, -sign, np.where(rng.integers(0, 2, (m + block - 1) // block).repeat(block)[:m], 1, -1)):
            rows.append(np.repeat((s * h)[:, None], 8, axis=1))
            rows.append(s[:, None] * rng.integers(h - 40, h + 1, (m, 8)))
        block *= 2
    for v in range(h - 24, h + 1):  # the same value in every ring, both signs
        rows += [np.full((m, 8), v), np.full((m, 8), -v)]
    for _ in range(64):
        v = rng.integers(-h, h + 1, 8)
        rows.append(np.repeat(v[None], m, axis=0))
    # the products come out times -2^-32
    vals = np.stack(rows).astype(np.int64)
    return vals * int(-(1 << 32) % q) % q


def test_inverse_of_the_patterns():
    """The chosen polynomials have the chosen residues (one prime, both rings)."""
    q, n = 18433, 256
    rng = np.random.default_rng(5)
    vals = rng.integers(0, q, (2, n // 8, 8))
    for cyclic in (False, True):
        a = _inverse(vals, q, n, cyclic)
        m = n // 8
        psi = _root(q, m if cyclic else 2 * m)
        for ring in (0, 1, 5, m - 1):
            # ring 2 i or 2 i + 1 is x^8 - z or x^8 + z for the last level's root z
            g = ring // 2
            e = _bitrev(g, m.bit_length() - 1) // 2 if cyclic else _bitrev(m // 2 + g, m.bit_length() - 1)
            z = pow(psi, e, q) * (-1 if ring & 1 else 1) % q
            p = np.array([pow(z, i, q) for i in range(n // 8)], dtype=np.int64)
            got = (a.reshape(2, n // 8, 8) * p[None, :, None] % q).sum(1) % q
            assert np.array_equal(got, vals[:, ring] % q)


@pytest.mark.gpu
@pytest.mark.parametrize("cyclic", [False, True])
@pytest.mark.parametrize("n", [256, 512, 1024])
def test_largest_sums_of_the_inverse(n, cyclic):
    from paper_2307_06554_gb300 import polymul as pm
    rng = np.random.default_rng(n)
    flags = pm.FLAG_CYCLIC if cyclic else 0
    qs = _primes(n if cyclic else 2 * n, 12000)
    assert 18433 in qs or cyclic
    for q in qs:
        a = _inverse(_patterns(q, n, rng), q, n, cyclic).astype(np.uint32)[:, None, :]
        one = np.zeros_like(a)
        one[:, :, 0] = 1
        with pm.Plan(n, [q], path=pm.PATH_NTT, flags=flags) as plan:
            plan.select(0)  # the unit, whatever the batch
            assert np.array_equal(run_plan_batch(plan, a, one), a), q
            assert np.array_equal(run_plan_batch(plan, one, a), a), q


@pytest.mark.gpu
@pytest.mark.parametrize("cyclic", [False, True])
def test_largest_sums_shared_operand(cyclic):
    import torch
    from paper_2307_06554_gb300 import polymul as pm
    n = 1024
    rng = np.random.default_rng(n + 1)
    for q in _primes(n if cyclic else 2 * n, 12000):
        b = _inverse(_patterns(q, n, rng), q, n, cyclic).astype(np.uint32)[:, None, :]
        a = np.zeros((1, n), np.uint32)
        a[0, 0] = 1
        with pm.Plan(n, [q], path=pm.PATH_NTT, flags=pm.FLAG_CYCLIC if cyclic else 0) as plan:
            ta, tb = (torch.from_numpy(x.view(np.int32)).cuda() for x in (a, b))
            tc = torch.full_like(tb, -1)
            pm.polymul_batch_shared(plan.handle, ta, tb, tc, len(b))
            torch.cuda.synchronize()
            assert np.array_equal(tc.cpu().numpy().view(np.uint32), b), q
