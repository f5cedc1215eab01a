"""Several host threads at once, each on its own stream and system: the tensor-core
reduction launches kernels whose shared memory depends on the system, and the limit
of a kernel's dynamic shared memory is shared by all threads of the process.  Every
reduction succeeds and gives the bits it gives alone."""
import threading

import pytest
import torch

import workloads as W
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu


def test_reductions_of_different_sizes_in_threads():
    from paper_1708_06290_gb300 import ssv
    sizes = [(600, 4, 12), (1500, 32, 6), (300, 16, 20), (900, 64, 8)]
    data, alone = [], []
    for n, m, _ in sizes:
        sysr = W.random_system(n, m, 2, seed=7300 + n)
        data.append((dev(sysr.A), dev(sysr.B), dev(sysr.C)))
        h = ssv.reduce(*data[-1], arith="tensor")
        alone.append([t.clone() for t in h.reduced()])
        h.close()
    torch.cuda.synchronize()
    bad = []

    def work(k):
        st = torch.cuda.Stream()
        for _ in range(sizes[k][2]):
            try:
                with torch.cuda.stream(st):
                    h = ssv.reduce(*data[k], arith="tensor", stream=st)
                    got = h.reduced(stream=st)
                    st.synchronize()
                    if not all(torch.equal(a, b) for a, b in zip(got, alone[k])):
                        bad.append((sizes[k], "other bits"))
                    h.close()
            except Exception as e:  # noqa: BLE001 - reported by the main thread
                bad.append((sizes[k], str(e)))

    ts = [threading.Thread(target=work, args=(k,)) for k in range(len(sizes))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad, bad[:4]
