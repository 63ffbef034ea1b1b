"""One context per host thread, contexts of different shapes at once.

The contraction and pack kernels are launched with a shared-memory size that
depends on the bins, one kernel for several sizes, and a kernel's limit is one
for all threads: a thread that set it to its own smaller size between another
thread's call and its launch made that launch fail.  Two threads compute
with 10 and with 20 bins side by side; every result is the one that the
context gives alone."""
import threading

import numpy as np
import pytest

from paper_2604_08855_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["FP32", "BF16X3"])
def test_contexts_of_two_shapes_in_two_threads(prec):
    torch = pytest.importorskip("torch")
    from paper_2604_08855_gb300 import build
    build.build()
    from paper_2604_08855_gb300 import ctb
    xyz, w = synth.thomas(400, 300.0, 4, 5.0, seed=95)
    start = threading.Barrier(2)
    out = {}

    def work(nbins):
        try:
            stream = torch.cuda.Stream()
            est = ctb.CTB(300.0, 2.0, 40.0, nbins, 10)
            est.set_stream(stream)
            est.set_option(ctb.OPT_PRECISION, getattr(ctb, "PREC_" + prec))
            est.set_points(xyz, w)
            first = est.compute()
            start.wait(60)
            for _ in range(3000):
                if not np.array_equal(est.compute(), first):
                    raise AssertionError("another thread changed the result")
            est.close()
            out[nbins] = "ok"
        except Exception as e:  # noqa: BLE001 -- reported below
            out[nbins] = repr(e)
            start.abort()

    threads = [threading.Thread(target=work, args=(nb,)) for nb in (10, 20)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert out == {10: "ok", 20: "ok"}
