"""Kernels that store into other CTAs' shared memory pass a cluster barrier
first: a CTA of the cluster that has not started may not be accessed.  Read
from the source, since a run cannot show the order in which CTAs start; the
GPU test then runs every cluster kernel of a plan once and twice per cluster."""
import os
import re

import numpy as np
import pytest

from oracle import native
from paper_2307_06554_gb300 import workloads as wl
from paper_2307_06554_gb300.build import CSRC

from helpers import assert_equal_residues, run_plan_batch

# calls through which a kernel reaches other CTAs' shared memory
REMOTE = r"\b(?:cfwd|cinv|cstore|cload|fwd_db|inv_db|fwd_from|inv_from)\s*<"


def _kernel_bodies():
    """(name, body) of every __global__ function of the cluster file, comments removed."""
    with open(os.path.join(CSRC, "ntt_cluster.cu")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    out = []
    for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\([^{;]*\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        out.append((m.group(1), text[m.end():i]))
    return out


def test_a_barrier_precedes_the_first_remote_access():
    bodies = _kernel_bodies()
    assert {name for name, _ in bodies} == {"k_ntt_cluster", "k_ntt_cluster2"}
    for name, body in bodies:
        first = re.search(REMOTE, body).start()
        loop = re.search(r"\bfor \(uint64_t u = cluster_id", body).start()
        arrive, wait = body.find("cluster_start_arrive();"), body.find("cluster_start_wait();")
        assert 0 <= arrive < wait < loop < first, name
        assert "ClusterSync{}()" not in body[:wait], name  # no other cluster barrier in between


@pytest.mark.gpu
@pytest.mark.parametrize("n,bits,dtype", [(8192, 61, np.uint64), (16384, 61, np.uint64), (16384, 31, np.uint32),
                                          (16384, 30, np.uint32)])
def test_cluster_kernels(n, bits, dtype):
    from paper_2307_06554_gb300 import polymul as pm
    rng = np.random.default_rng(n + bits)
    qs = wl.draw_primes(rng, 1, bits, bits, n.bit_length())
    a = wl.uniform_coeffs(rng, 90, qs, n, dtype)
    b = wl.uniform_coeffs(rng, 90, qs, n, dtype)
    idx = [0, 47, 89]
    want = native.polymul_batch(a[idx], b[idx], qs)
    with pm.Plan(n, qs, path=pm.PATH_NTT) as plan:
        for c in range(plan.info["candidates"]):
            plan.select(c)
            assert_equal_residues(run_plan_batch(plan, a, b)[idx], want, "candidate %d" % c)
