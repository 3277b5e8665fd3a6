"""Which of the server's streams a request takes (serve_queue.h, on the host),
and page-locked and pageable requests mixed on one server."""
import subprocess

import numpy as np
import pytest

from oracle import native
from paper_2307_06554_gb300 import workloads as wl
from paper_2307_06554_gb300.build import CSRC

HOST = r"""
#include <cstdio>
#include "serve_queue.h"
using pm::ServeQueues;
static int bad = 0;
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); bad = 1; } } while (0)
constexpr uint64_t MB = 1 << 20;
int main() {
  ServeQueues s;
  // staged requests alone: the lane with the least bytes in flight
  s.reset(2);
  CHECK(s.admit(false, 9 * MB) == 0);
  CHECK(s.admit(false, 2 * MB) == 1);
  CHECK(s.admit(false, 3 * MB) == 1);
  CHECK(s.admit(false, 5 * MB) == 1);
  CHECK(s.admit(false, MB) == 0);
  s.release(0, false, 9 * MB);
  CHECK(s.admit(false, MB) == 0);
  // direct requests alone: lanes first, then, from half a MB, the other streams
  s.reset(2);
  CHECK(s.admit(true, MB) == 0);
  CHECK(s.admit(true, MB) == 1);
  CHECK(s.admit(true, MB) == 2);
  CHECK(s.admit(true, MB) == 3);
  CHECK(s.admit(true, MB / 4) == 0);  // a small one stays on a lane
  s.release(2, true, MB);
  CHECK(s.load(2) == 0 && s.load(3) == MB);
  // a large staged request occupies its copy streams too: a direct one takes
  // none of them while another lane's are idle
  s.reset(2);
  CHECK(s.admit(false, 100 * MB) == 0);
  CHECK(s.admit(true, MB) == 1);
  CHECK(s.admit(true, MB) == 3);  // lane 1's copy-in stream, not lane 0's
  CHECK(s.admit(true, MB) == 5);  // lane 1's copy-out stream
  // and a staged request stays off a lane whose copy streams run large direct kernels
  s.reset(2);
  CHECK(s.admit(true, 2 * MB) == 0);
  CHECK(s.admit(true, 3 * MB) == 1);
  CHECK(s.admit(true, 90 * MB) == 2);  // lane 0's copy-in stream
  CHECK(s.admit(false, MB) == 1);
  // everything released: no load is left
  s.release(0, true, 2 * MB);
  s.release(1, true, 3 * MB);
  s.release(2, true, 90 * MB);
  s.release(1, false, MB);
  for (int q = 0; q < s.queues(); ++q) CHECK(s.load(q) == 0);
  return bad;
}
"""


def test_queue_choice(tmp_path):
    src, exe = tmp_path / "queues.cpp", tmp_path / "queues"
    src.write_text(HOST)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


HOST_SMALL = r"""
#include "serve_queue.h"
int main() {
  pm::ServeQueues s;
  s.reset(2);
  // below a MB a direct request stays on a lane while the lanes have less than
  // 2 MB ahead, below half a MB always
  for (int i = 0; i < 6; ++i)
    if (s.admit(true, 768 << 10) >= 2) return 1;
  if (s.admit(true, 256 << 10) >= 2) return 1;
  if (s.occupied() != 2) return 2;
  const int r = s.admit(true, 768 << 10);
  if (r < 2) return 4;
  s.release(r, true, 768 << 10);
  // the queues past the lanes are looked at only while one holds a request
  const int q = s.admit(true, 2 << 20);
  if (q < 2 || s.occupied() != 6) return 3;
  s.release(q, true, 2 << 20);
  return s.occupied() != 2;
}
"""


def test_small_requests_keep_to_the_lanes(tmp_path):
    src, exe = tmp_path / "small.cpp", tmp_path / "small"
    src.write_text(HOST_SMALL)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)])
    assert subprocess.run([str(exe)]).returncode == 0


@pytest.mark.gpu
@pytest.mark.parametrize("bits", [59, 61])
def test_mixed_routes(bits):
    """Large page-locked (direct) and pageable (staged) requests in turn on two
    lanes: the two routes agree, and samples agree with the oracle.  61-bit
    primes take the Harvey-bound kernels, 59-bit ones those of small words."""
    import torch
    from paper_2307_06554_gb300 import polymul as pm
    rng = np.random.default_rng(90 + bits)
    pool = wl.draw_primes(rng, 6, bits, bits, 17)
    degrees = (16, 512, 4096, 8192, 16384, 32768)
    reqs = []
    for i in range(30):
        n = degrees[i % len(degrees)]
        idx = np.sort(rng.permutation(6)[:1 + i % 4]).astype(np.uint32)
        qs = [pool[j] for j in idx]
        reqs.append((n, idx, qs, wl.uniform_coeffs(rng, 1, qs, n, np.uint64)[0],
                     wl.uniform_coeffs(rng, 1, qs, n, np.uint64)[0]))

    def pinned(x):
        return torch.from_numpy(x.view(np.int64)).pin_memory().numpy().view(np.uint64)

    with pm.Server(pool, 32768, device_bytes=1 << 28, lanes=2) as srv:
        tickets, outs = [], []
        for n, idx, qs, a, b in reqs:
            pair = []
            for conv in (pinned, np.copy):  # direct, staged
                xa, xb, c = conv(a), conv(b), conv(np.zeros_like(a))
                pair.append(c)
                tickets.append((srv.submit(n, idx, xa, xb, c), xa, xb))
            outs.append(pair)
        for t, *_ in tickets:
            srv.wait(t)
        st = srv.stats()
    assert st["completed"] == 60 and st["completed_direct"] == 30
    for i, (n, idx, qs, a, b) in enumerate(reqs):
        assert np.array_equal(outs[i][0], outs[i][1]), i
        if n <= 8192 and i < 12:
            assert np.array_equal(outs[i][0], native.polymul_batch(a[None], b[None], qs)[0]), i
