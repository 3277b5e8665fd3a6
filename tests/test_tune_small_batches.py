"""Tuning that settles on the default kernel keeps the kernel of small batches.
Which kernel a batch runs is read from a captured graph (grid and block of its
one kernel node); a cache file makes the tuned choice certain."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2307_06554_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import ctypes, json, sys
sys.path.insert(0, %r)
import torch
from paper_2307_06554_gb300 import polymul

class KernelNode(ctypes.Structure):  # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p)] + [(f, ctypes.c_uint) for f in
        ("gx", "gy", "gz", "bx", "by", "bz", "smem")] + [(f, ctypes.c_void_p) for f in
        ("params", "extra", "kern", "ctx")]

cu = ctypes.CDLL("libcuda.so.1")
def ok(r):
    assert r == 0, r

def shape(plan, batch):
    # grid and block of the one kernel that a batch launches
    a = torch.zeros(batch, plan.info["k"], plan.info["n"], dtype=torch.int64, device="cuda")
    b, c = torch.zeros_like(a), torch.zeros_like(a)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    s = ctypes.c_void_p(st.cuda_stream)
    ok(cu.cuStreamBeginCapture_v2(s, 2))
    plan.batch(a, b, c, stream=st.cuda_stream)
    g = ctypes.c_void_p()
    ok(cu.cuStreamEndCapture(s, ctypes.byref(g)))
    cnt = ctypes.c_size_t(8)
    nodes = (ctypes.c_void_p * 8)()
    ok(cu.cuGraphGetNodes(g, nodes, ctypes.byref(cnt)))
    assert cnt.value == 1
    kp = KernelNode()
    ok(cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(nodes[0]), ctypes.byref(kp)))
    ok(cu.cuGraphDestroy(g))
    return [kp.gx, kp.bx, kp.smem]

n, qs, tune = json.loads(sys.argv[1])
out = {}
with polymul.Plan(n, qs, path=polymul.PATH_NTT) as p:
    out["untuned"] = shape(p, 1)
    out["default"] = p.select(0)
    out["selected"] = shape(p, 1)
    out["other"] = p.select(p.info["candidates"] - 1)
    p.tune(tune)
    out["chosen"] = p.info
    out["tuned"] = shape(p, 1)
    p.select(0)
    out["reselected"] = shape(p, 1)
print(json.dumps(out))
""" % ROOT


def _run(n, qs, tune, cache):
    r = subprocess.run([sys.executable, "-c", SCRIPT, json.dumps([n, qs, tune])], capture_output=True, text=True,
                       env=dict(os.environ, POLYMUL_TUNE_CACHE=str(cache)))
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def _label(info):
    return "ntt-rb%d-m%d-r%d-p%d-o%d-b%d-s%d" % tuple(
        info[f] for f in ("radix_bits", "ntt_mode", "regs", "exchange_pad", "one_operand", "block", "smem_bytes"))


def test_default_kernel_keeps_its_small_form(tmp_path):
    n, qs = 32768, wl.draw_primes(np.random.default_rng(1), 1, 59, 59, 16)
    cache = tmp_path / "tune.txt"
    first = _run(n, qs, 64, cache)
    assert first["untuned"] != first["selected"]  # small batches have a kernel of their own
    key = cache.read_text().split("\t")[0]
    # the default kernel is the choice for 64 products
    cache.write_text("%s\t%s\n" % (key, _label(first["default"])))
    got = _run(n, qs, 64, cache)
    assert got["chosen"]["tuned"] == 1 and got["chosen"]["regs"] == got["default"]["regs"]
    assert got["tuned"] == got["untuned"] and got["reselected"] == got["selected"]
    # another candidate is: it runs whatever the batch
    cache.write_text("%s\t%s\n" % (key, _label(first["other"])))
    got = _run(n, qs, 64, cache)
    assert got["chosen"]["block"] == got["other"]["block"] and got["chosen"]["smem_bytes"] == got["other"]["smem_bytes"]
    # the default kernel measured at a batch as small as that, and kept: it runs there
    cache.write_text("%sb8\t%s\n" % (key[:-3], _label(first["default"])))
    assert _run(n, qs, 8, cache)["tuned"] == got["selected"]
