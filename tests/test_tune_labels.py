"""A stored tuning choice names one candidate: with a cache file that holds a
different candidate of a plan for each batch bucket, a fresh process takes
exactly those kernels, also where several share their radix or are clusters;
labels that name no candidate are measured again."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2307_06554_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHAPE = ("radix_bits", "ntt_mode", "regs", "exchange_pad", "one_operand", "block", "smem_bytes")

SCRIPT = """
import sys, json
sys.path.insert(0, %r)
from paper_2307_06554_gb300 import polymul
n, qs, batches = json.loads(sys.argv[1])
p = polymul.Plan(n, qs, path=polymul.PATH_NTT)
out = []
for b in batches:
    p.tune(b)
    out.append(p.info)
print(json.dumps(out))
""" % ROOT


def _tuned(cache, n, qs, batches):
    r = subprocess.run([sys.executable, "-c", SCRIPT, json.dumps([n, qs, batches])], capture_output=True, text=True,
                       env=dict(os.environ, POLYMUL_TUNE_CACHE=str(cache)), check=True)
    return json.loads(r.stdout.strip().splitlines()[-1])


def _label(info):
    return "ntt-rb%d-m%d-r%d-p%d-o%d-b%d-s%d" % tuple(info[f] for f in SHAPE)


@pytest.mark.parametrize("n,bits", [(4096, 30), (16384, 30), (4096, 59), (32768, 59)])
def test_each_label_brings_back_its_candidate(tmp_path, n, bits):
    from paper_2307_06554_gb300 import polymul as pm
    qs = wl.draw_primes(np.random.default_rng(n), 1, bits, bits, n.bit_length())
    with pm.Plan(n, qs, path=pm.PATH_NTT) as plan:
        infos = [plan.select(i) for i in range(plan.info["candidates"])]
    assert len(infos) >= 2
    cache = tmp_path / "tune.txt"
    _tuned(cache, n, qs, [1])
    key, label = cache.read_text().strip().split("\t")
    assert label in [_label(i) for i in infos] and key.endswith("|b1")
    batches = [1 << i for i in range(len(infos))]
    cache.write_text("".join("%s|b%d\t%s\n" % (key[:-3], b, _label(i)) for b, i in zip(batches, infos)))
    before = cache.read_text()
    got = _tuned(cache, n, qs, batches)
    assert [[g[f] for f in SHAPE] for g in got] == [[i[f] for f in SHAPE] for i in infos]
    assert cache.read_text() == before  # every choice came from the file


def test_unknown_label_is_measured_again(tmp_path):
    cache = tmp_path / "tune.txt"
    _tuned(cache, 1024, [12289], [64])
    key, _ = cache.read_text().strip().split("\t")
    cache.write_text("%s\tntt-rb4\n" % key)
    _tuned(cache, 1024, [12289], [64])
    lines = cache.read_text().strip().splitlines()
    assert len(lines) == 2 and lines[1].split("\t")[1] != "ntt-rb4"
