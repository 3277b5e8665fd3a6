"""Plans with POLYMUL_FLAG_OVERLAP take the kernels of overlapped batches only
for batches that may start before their predecessor has finished: not for the
first on a stream, nor for one that reads its predecessor's result.  Read from a
captured stream's kernel nodes (block and shared memory of each launch)."""
import ctypes

import numpy as np
import pytest

from paper_2307_06554_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


class KernelNode(ctypes.Structure):  # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = ([("func", ctypes.c_void_p)]
                + [(f, ctypes.c_uint) for f in ("gx", "gy", "gz", "bx", "by", "bz", "smem")]
                + [(f, ctypes.c_void_p) for f in ("params", "extra", "kern", "ctx")])


def _launches(stream, calls):
    """(block, shared memory) of the kernels that the calls launch, in launch order."""
    cu = ctypes.CDLL("libcuda.so.1")

    def ok(r):
        assert r == 0, r

    s, g = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    out = []
    ok(cu.cuStreamBeginCapture_v2(s, 2))
    for call in calls:
        call()
    ok(cu.cuStreamEndCapture(s, ctypes.byref(g)))
    count, nodes = ctypes.c_size_t(16), (ctypes.c_void_p * 16)()
    ok(cu.cuGraphGetNodes(g, nodes, ctypes.byref(count)))
    for i in range(count.value):
        kp = KernelNode()
        ok(cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(nodes[i]), ctypes.byref(kp)))
        out.append((kp.bx, kp.smem))
    ok(cu.cuGraphDestroy(g))
    return out


# n, bits, products, the shape of the kernel of batches that run ahead
@pytest.mark.parametrize("n,bits,batch,shape", [
    (8192, 30, 200, {"radix_bits": 4, "exchange_pad": 0, "regs": 128}),
    (8192, 31, 350, {"radix_bits": 4, "exchange_pad": 0, "regs": 128}),
    (4096, 30, 800, {"radix_bits": 4, "exchange_pad": 0, "regs": 128}),
])
def test_kernel_by_dependence(n, bits, batch, shape):
    import torch
    from paper_2307_06554_gb300 import polymul as pm
    qs = wl.draw_primes(np.random.default_rng(n), 1, bits, bits, n.bit_length())
    a, b, c, d, e = (torch.zeros(batch, 1, n, dtype=torch.int32, device="cuda") for _ in range(5))
    st = torch.cuda.Stream()
    with pm.Plan(n, qs, path=pm.PATH_NTT, flags=pm.FLAG_OVERLAP) as probe:
        infos = [probe.select(i) for i in range(probe.info["candidates"])]
    kernel = lambda i: (i["block"], i["smem_bytes"])  # noqa: E731
    default = kernel(infos[0])
    ahead = [kernel(i) for i in infos if all(i[k] == v for k, v in shape.items())]
    assert len(ahead) == 1 and ahead[0] != default
    for flags, second in ((pm.FLAG_OVERLAP, ahead[0]), (0, default)):
        with pm.Plan(n, qs, path=pm.PATH_NTT, flags=flags) as plan:
            torch.cuda.synchronize()
            plan.batch(a, b, e, stream=torch.cuda.current_stream().cuda_stream)  # another stream's record
            torch.cuda.synchronize()
            got = _launches(st, [
                lambda: plan.batch(a, b, c, stream=st.cuda_stream),  # the first on the stream
                lambda: plan.batch(a, b, d, stream=st.cuda_stream),  # independent of it
                lambda: plan.batch(d, b, e, stream=st.cuda_stream),  # reads its result
            ])
        if flags == 0:
            assert got == [default] * 3
        else:
            # the stream's handle may have carried a launch of an earlier stream object
            assert got[0] in (default, ahead[0]) and got[1:] == [second, default], got
