"""The work this library is measured on: exact products in Z_q[x]/(x^n + 1)
through its public entry points, over the sizes its users run.

Sizes come from the five standing workloads of
``paper_2307_06554_gb300/workloads.py`` (ring_small, ring_1024, rns_4096,
ragged_2000, serve_20k), from the benchmark's tensor and shared-operand legs,
and from generic degrees between and beyond them.  ``listed()`` says beside
each case what it stands for; ``draw(rng)`` draws from the same kinds over
their whole ranges.
"""
import ctypes
import math
import random

import numpy as np
import torch

from paper_2307_06554_gb300 import polymul, workloads


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest ring in use (a Kyber-sized ring whose modulus has no
        # 2n-th root of unity): one product's latency and the launch
        dict(name="ring_small", kind="batch", n=256, k=1, bits=0, q=3329, batch=64, overlap=False, ternary=False,
             cyclic=False),
        # the headline: NTRU/Falcon-sized ring, thousands of products back to
        # back on one stream, batches allowed to overlap
        dict(name="ring_1024", kind="batch", n=1024, k=1, bits=0, q=12289, batch=4096, overlap=True, ternary=False,
             cyclic=False),
        # RNS products of a homomorphic-encryption ring: eight 30-bit primes,
        # a uniform, b ternary
        dict(name="rns_4096", kind="batch", n=4096, k=8, bits=30, q=0, batch=256, overlap=False, ternary=True,
             cyclic=False),
        # a large degree at an odd batch with 31-bit primes (the widest
        # 32-bit words): 111 rows, fewer than the SMs of the device
        dict(name="odd_16384", kind="batch", n=16384, k=3, bits=31, q=0, batch=37, overlap=False, ternary=False,
             cyclic=False),
        # 64-bit words at a moderate degree (two 59-bit primes)
        dict(name="words64_4096", kind="batch", n=4096, k=2, bits=59, q=0, batch=128, overlap=False, ternary=False,
             cyclic=False),
        # 64-bit words at a bootstrapping degree: the thread-block-cluster
        # kernels
        dict(name="words64_32768", kind="batch", n=32768, k=8, bits=59, q=0, batch=16, overlap=False, ternary=False,
             cyclic=False),
        # 2000 products of uneven degree and prime count, prepared once and
        # replayed as a graph
        dict(name="uneven_2000", kind="uneven", count=2000, kmax=16, pool=64, lo=10, hi=14, shape=4),
        # one public polynomial against a batch (keys, matrices of a scheme)
        dict(name="shared_1024", kind="shared", n=1024, k=1, bits=0, q=12289, batch=4096, cyclic=False),
        # the matrix form on the tensor cores, the paper's own question: two
        # digits of 8 bits
        dict(name="tensor_1024", kind="tensor", n=1024, k=1, bits=0, q=12289, batch=4096, ternary=False),
        # the matrix form at full 30-bit moduli: four digits a side, K chunks
        # drained into 64-bit sums
        dict(name="tensor_4096", kind="tensor", n=4096, k=8, bits=30, q=0, batch=64, ternary=False),
        # operands and results in page-locked host memory, one synchronous call
        dict(name="host_1024", kind="host", n=1024, k=1, bits=0, q=12289, batch=4096),
        # the request server: mixed degrees and prime counts of 59 bits from
        # page-locked host buffers, all queued at once
        dict(name="serve_mix", kind="serve", count=200, kmax=8, pool=8, lo=12, hi=14, lanes=8, shape=5),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _spread(rng, cost, least, most):
    """A batch whose work (batch * cost) is spread over [least, most] on a
    logarithmic scale; odd values as likely as even ones."""
    lo = max(1, -(-least // cost))
    hi = max(lo, most // cost)
    return _log_int(rng, lo, hi)


def _small_bits(rng, n, most):
    """A width from the smallest up to `most` bits that has a prime
    q = 1 mod 2n."""
    return rng.choice([w for w in range(n.bit_length() + 1, most + 1)
                       if any(workloads.is_prime(1 + 2 * n * j)
                              for j in range((1 << (w - 1)) // (2 * n), ((1 << w) - 2) // (2 * n) + 1))])


def draw(rng):
    kind = rng.choice(["batch", "batch", "batch", "batch", "aux", "words64", "words64", "uneven", "shared", "tensor",
                       "host", "serve"])
    coin = lambda p: rng.random() < p  # noqa: E731
    if kind == "batch":  # 32-bit words, own primes
        n = 1 << rng.randint(8, 14)
        if coin(0.4):
            k, bits, q = 1, _small_bits(rng, n, 20), 0
        else:
            k, bits, q = rng.randint(1, 8), rng.randint(28, 31), 0
        return dict(kind="batch", n=n, k=k, bits=bits, q=q, batch=_spread(rng, n * k, 1 << 14, 1 << 23),
                    overlap=coin(0.4), ternary=coin(0.3), cyclic=coin(0.2))
    if kind == "aux":  # moduli without a root of unity
        n, q = rng.choice([(128, 3329), (256, 3329), (256, 4099), (512, 2053), (1024, 1031)])
        return dict(kind="batch", n=n, k=1, bits=0, q=q, batch=_log_int(rng, 1, 4096), overlap=coin(0.3),
                    ternary=coin(0.3), cyclic=False)
    if kind == "words64":
        n = 1 << rng.randint(10, 16)
        k = rng.randint(1, 8 if n < 65536 else 4)
        return dict(kind="batch", n=n, k=k, bits=rng.randint(50, 60), q=0,
                    batch=_spread(rng, n * k, 1 << 16, 1 << 22), overlap=coin(0.3), ternary=False, cyclic=coin(0.2))
    if kind == "uneven":
        lo = rng.randint(10, 12)
        return dict(kind="uneven", count=_log_int(rng, 50, 1500), kmax=rng.randint(1, 16), pool=rng.randint(16, 48),
                    lo=lo, hi=rng.randint(lo, 14), shape=rng.randrange(1 << 30))
    if kind == "shared":
        n = 1 << rng.randint(10, 13)
        k, bits = (1, _small_bits(rng, n, 17)) if coin(0.5) else (rng.randint(1, 4), rng.randint(28, 31))
        return dict(kind="shared", n=n, k=k, bits=bits, q=0, batch=_spread(rng, n * k, 1 << 14, 1 << 22),
                    cyclic=coin(0.2))
    if kind == "tensor":
        n = 1 << rng.randint(8, 12)
        k, bits = (1, _small_bits(rng, n, 17)) if coin(0.5) else (rng.randint(1, 4), rng.randint(28, 30))
        return dict(kind="tensor", n=n, k=k, bits=bits, q=0, batch=_spread(rng, n * n * k, 1 << 26, 1 << 32),
                    ternary=coin(0.3))
    if kind == "host":
        n = 1 << rng.randint(8, 13)
        k, bits = rng.choice([(1, _small_bits(rng, n, 20)), (3, 30), (2, 59)])
        return dict(kind="host", n=n, k=k, bits=bits, q=0, batch=_spread(rng, n * k, 1 << 14, 1 << 21))
    lo = rng.randint(10, 13)
    return dict(kind="serve", count=_log_int(rng, 20, 200), kmax=rng.randint(1, 8), pool=8, lo=lo,
                hi=rng.randint(lo, 14), lanes=8, shape=rng.randrange(1 << 30))


# ------------------------------------------------- moduli and lists of a case
def _moduli(case):
    if case["q"]:
        return [case["q"]]
    two_adic = case["n"].bit_length()  # q = 1 mod 2n
    return workloads.draw_primes(np.random.default_rng(1000 + case["bits"]), case["k"], case["bits"], case["bits"],
                                 two_adic)


def _pool(case):
    if case["kind"] == "uneven":
        return workloads.draw_primes(np.random.default_rng(case["shape"]), case["pool"], 28, 31, 15)
    return workloads.draw_primes(np.random.default_rng(case["shape"]), case["pool"], 59, 59, case["hi"] + 1)


def _products(case):
    """(n, prime indices) of each product of an uneven list or request mix;
    the list's shape belongs to the case, the coefficients to the seed."""
    rng = random.Random(case["shape"])
    out = []
    for _ in range(case["count"]):
        n = 1 << rng.randint(case["lo"], case["hi"])
        out.append((n, sorted(rng.sample(range(case["pool"]), rng.randint(1, min(case["kmax"], case["pool"]))))))
    return out


def _words64(case):
    return case["kind"] == "serve" or case.get("bits", 0) > 31


# ------------------------------------------------------------------- operands
def _uniform(gen, rows, n, q_rows, dtype):
    """[rows][n] values uniform in [0, q_rows[row])."""
    x = torch.randint(0, 1 << 62, (rows, n), generator=gen, device="cuda", dtype=torch.int64)
    return (x % q_rows.view(rows, 1)).to(dtype)


def _operands(case, seed):
    """a, b of a homogeneous case on the device, [batch][k][n] ([k][n] for a
    shared a)."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 2 + 1)
    qs = torch.tensor(_moduli(case), dtype=torch.int64, device="cuda")
    n, k, batch = case["n"], len(qs), case["batch"]
    dtype = torch.int64 if _words64(case) else torch.int32
    na = 1 if case["kind"] == "shared" else batch
    a = _uniform(gen, na * k, n, qs.repeat(na), dtype).view(na, k, n)
    if case.get("ternary"):  # one small polynomial per product, -1 lifted to q - 1
        t = torch.randint(-1, 2, (batch, 1, n), generator=gen, device="cuda", dtype=torch.int64)
        b = torch.where(t < 0, qs.view(1, k, 1) - 1, t).to(dtype).contiguous()
    else:
        b = _uniform(gen, batch * k, n, qs.repeat(batch), dtype).view(batch, k, n)
    return (a[0].contiguous() if case["kind"] == "shared" else a), b


def _flat_operands(case, seed):
    """Flat a, b of an uneven list or a request mix, products back to back,
    [k][n] each."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 2 + 1)
    pool = torch.tensor(_pool(case), dtype=torch.int64, device="cuda")
    rows_n, rows_p = [], []
    for n, idx in _products(case):
        rows_n += [n] * len(idx)
        rows_p += idx
    dtype = torch.int64 if _words64(case) else torch.int32
    rows_n = torch.tensor(rows_n, device="cuda")
    q = torch.repeat_interleave(pool[torch.tensor(rows_p, device="cuda")], rows_n)
    out = []
    for _ in range(2):
        x = torch.randint(0, 1 << 62, q.shape, generator=gen, device="cuda", dtype=torch.int64)
        out.append((x % q).to(dtype))
    return out


# ----------------------------------------------------------- prepare and run
_STREAM = None


def _stream():
    """The program's one working stream (a stream of its own: the default
    stream takes no overlapped batches)."""
    global _STREAM
    if _STREAM is None:
        _STREAM = torch.cuda.Stream()
    return _STREAM


class _State:
    """Inputs, output buffers and the handle of one case; the handle is closed
    with the state."""

    def __init__(self, kind):
        self.kind = kind
        self.owner = None

    def __del__(self):
        if self.owner is not None:
            self.owner.close()


def _pinned(x):
    h = torch.empty(x.shape, dtype=x.dtype, pin_memory=True)
    h.copy_(x)
    return h


def prepare(case, seed):
    s = _State(case["kind"])
    s.stream = _stream()
    if s.kind in ("batch", "tensor", "shared", "host"):
        a, b = _operands(case, seed)
        flags = 0
        if case.get("overlap"):
            flags |= polymul.FLAG_OVERLAP
        if case.get("cyclic"):
            flags |= polymul.FLAG_CYCLIC
        if s.kind == "tensor" and case["ternary"]:
            flags |= polymul.FLAG_TERNARY_B
        s.owner = polymul.Plan(case["n"], _moduli(case),
                               path=polymul.PATH_TENSOR if s.kind == "tensor" else polymul.PATH_AUTO, flags=flags)
        if s.kind == "host":
            s.a, s.b = _pinned(a), _pinned(b)
            s.c = torch.empty(b.shape, dtype=b.dtype, pin_memory=True)
        else:
            s.a, s.b, s.c = a, b, torch.empty_like(b)
    elif s.kind == "uneven":
        s.a, s.b = _flat_operands(case, seed)
        s.c = torch.empty_like(s.a)
        s.owner = polymul.Ragged(_pool(case), 1 << case["hi"], _products(case))
    else:
        a, b = _flat_operands(case, seed)
        s.a, s.b = _pinned(a), _pinned(b)
        s.c = torch.empty(a.shape, dtype=a.dtype, pin_memory=True)
        requests, off = [], 0
        for n, idx in _products(case):
            rows = slice(off, off + n * len(idx))
            requests.append((n, idx, s.a[rows], s.b[rows], s.c[rows]))
            off += n * len(idx)
        s.owner = polymul.Server(_pool(case), 1 << case["hi"], device_bytes=1 << 28, lanes=case["lanes"])
        s.requests = polymul.Server.prepare(requests)
        s.arrivals = (ctypes.c_double * len(requests))()
    torch.cuda.synchronize()
    return s


def run(s):
    if s.kind in ("batch", "tensor"):
        s.owner.batch(s.a, s.b, s.c, stream=s.stream)
    elif s.kind == "shared":
        polymul.polymul_batch_shared(s.owner.handle, s.a, s.b, s.c, s.b.shape[0], stream=s.stream)
    elif s.kind == "host":
        s.owner.batch_host(s.a, s.b, s.c)
    elif s.kind == "uneven":
        s.owner.run(s.a, s.b, s.c, stream=s.stream, graph=True)
    else:
        s.owner.replay(s.requests, s.arrivals)
    return s.c


# ----------------------------------------------------------------------- work
def _rows(case):
    """(n, rows) of a case: rows = (product, prime) pairs of degree n."""
    if case["kind"] in ("uneven", "serve"):
        rows = {}
        for n, idx in _products(case):
            rows[n] = rows.get(n, 0) + len(idx)
        return sorted(rows.items())
    return [(case["n"], case["batch"] * max(1, case["k"]))]


def work(case):
    """Operands read and results written once; for the matrix form also the
    2 n^2 operations of each pair of 8-bit digits."""
    word = 8 if _words64(case) else 4
    rows = _rows(case)
    coeffs = sum(n * r for n, r in rows)
    read = coeffs + (case["n"] * case["k"] if case["kind"] == "shared" else coeffs)
    flops = 0
    if case["kind"] == "tensor":
        digits = -(-(case["bits"] or case["q"].bit_length()) // 8)
        flops = sum(2 * n * n * r for n, r in rows) * digits * (1 if case["ternary"] else digits)
    return {"bytes": (read + coeffs) * word, "flops": flops}


# ---------------------------------------------------------------------- exact
def _exact_rows(a, b, q, cyclic):
    """Products of [rows][n] int64 tensors modulo the [rows] moduli q: balanced
    sums of small limbs through float64 transforms long enough for the whole
    product, rounded to integers and recombined modulo q."""
    rows, n = a.shape
    w = 11 if int(q.max()) < (1 << 33) else 12
    limbs = 3 if w == 11 else 6
    mask = (1 << w) - 1
    fa = [torch.fft.rfft(((a >> (w * i)) & mask).double(), 2 * n) for i in range(limbs)]
    fb = [torch.fft.rfft(((b >> (w * i)) & mask).double(), 2 * n) for i in range(limbs)]
    q = q.view(rows, 1)
    acc = torch.zeros_like(a)
    for e in range(2 * limbs - 2, -1, -1):
        f = sum(fa[i] * fb[e - i] for i in range(max(0, e - limbs + 1), min(e, limbs - 1) + 1))
        v = torch.fft.irfft(f, 2 * n).round().to(torch.int64)
        v = v[:, :n] + v[:, n:] if cyclic else v[:, :n] - v[:, n:]
        for _ in range(w):  # acc * 2^w mod q, one doubling at a time
            acc = acc * 2
            acc = torch.where(acc >= q, acc - q, acc)
        acc = (acc + v) % q  # the divisor's sign: in [0, q)
    return acc


def _exact_chunks(a, b, q, cyclic, most=1 << 21):
    out = torch.empty(b.shape, dtype=torch.int64, device=b.device)
    step = max(1, most // b.shape[1])
    for r in range(0, b.shape[0], step):
        out[r:r + step] = _exact_rows(a[r:r + step].long(), b[r:r + step].long(), q[r:r + step], cyclic)
    return out


def exact(case, seed):
    if case["kind"] in ("uneven", "serve"):
        a, b = _flat_operands(case, seed)
        pool = torch.tensor(_pool(case), dtype=torch.int64, device="cuda")
        c = torch.empty_like(a)
        by_degree, off = {}, 0
        for n, idx in _products(case):
            for i in idx:
                by_degree.setdefault(n, []).append((off, i))
                off += n
        for n, rows in by_degree.items():
            at = torch.tensor([r[0] for r in rows], device="cuda").view(-1, 1) + torch.arange(n, device="cuda")
            q = pool[torch.tensor([r[1] for r in rows], device="cuda")]
            c[at] = _exact_chunks(a[at], b[at], q, False).to(c.dtype)
        return c
    a, b = _operands(case, seed)
    n = case["n"]
    if case["kind"] == "shared":
        a = a.unsqueeze(0).expand(b.shape)
    q = torch.tensor(_moduli(case), dtype=torch.int64, device="cuda").repeat(b.shape[0])
    c = _exact_chunks(a.reshape(-1, n), b.reshape(-1, n), q, bool(case.get("cyclic")))
    return c.to(b.dtype).view(b.shape)
