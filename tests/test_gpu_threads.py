"""Contexts of different orders on two threads: the tensor-core kernels' shared-memory size differs with the
order, and neither thread's launches may depend on what the other last asked for.

Reference: the same evaluations one after the other, bit for bit (every sum has one order).
"""
import threading

import pytest
import torch

from synth import charges, cube_points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,depth", [("fp32", 3), ("fp16x3", 3), ("bf16x6", 3)])
def test_two_orders_on_two_threads(precision, depth):
    import paper_2604_19243_gb300 as pkg
    n, rounds = 2001, 300
    x, q = torch.from_numpy(cube_points(n)).cuda(), torch.from_numpy(charges(n, "u11")).cuda()
    torch.cuda.synchronize()
    f, want, failed, streams = [], [], [], [torch.cuda.Stream() for _ in range(2)]
    for p, s in zip((3, 6), streams):   # a context keeps the stream that it was made on
        with torch.cuda.stream(s):
            f.append(pkg.FMM(p=p, depth=depth, precision=precision, domain=((0.0, 0.0, 0.0), 1.0)).build_tree(x).precompute())
            want.append(f[-1].evaluate(q))
    torch.cuda.synchronize()

    def work(k):
        try:
            with torch.cuda.stream(streams[k]):
                for _ in range(rounds):
                    got = f[k].evaluate(q)
                torch.cuda.synchronize()
            if not all(torch.equal(a, b) for a, b in zip(got, want[k])):
                failed.append((k, "values"))
        except Exception as e:   # to the main thread
            failed.append((k, repr(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for c in f:
        c.sync()
