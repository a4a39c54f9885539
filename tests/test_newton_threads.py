"""Newton steps of several sizes from several host threads at once, each on its
own handle and stream: handles are independent of each other."""
import threading

import numpy as np
import pytest

import synth

from test_newton_int import linear_plus_square

pytestmark = pytest.mark.gpu


def test_sizes_from_several_threads():
    """Systems whose eliminations need different amounts of shared memory
    (51 to 220 KiB), 1500 steps each: every call is accepted, and every thread ends with
    the bits that one thread alone gets."""
    import torch

    import paper_1201_0499_gb300 as pkg

    sizes = (36, 60, 77)

    def steps(n, count, out):
        try:
            ev = pkg.PolyEval(linear_plus_square(750, n), pkg.PE_DD, max_points=1)
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                x0 = torch.from_numpy(synth.points(751, n, 1)).cuda()
                f = torch.empty((n, 1, 4), dtype=torch.float64, device="cuda")
                J = torch.empty((n, n, 1, 4), dtype=torch.float64, device="cuda")
                norms = torch.empty((1, 2), dtype=torch.float64, device="cuda")
                for i in range(count):
                    x = x0.clone()
                    pkg.polyeval_newton(ev.handle, x, 1, f, J, norms, stream.cuda_stream)
                    if i % 50 == 0:
                        stream.synchronize()
                stream.synchronize()
                out[n] = x.cpu().numpy()
            ev.close()
        except pkg.PolyEvalError as e:
            out[n] = e

    alone, together = {}, {}
    for n in sizes:
        steps(n, 1, alone)
    threads = [threading.Thread(target=steps, args=(n, 1500, together)) for n in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for n in sizes:
        assert isinstance(together[n], np.ndarray), (n, together[n])
        assert np.array_equal(alone[n], together[n])
