"""Contexts of their own in two threads: the size of one launch is no other's
business."""
import threading

import numpy as np
import pytest

from paper_2311_16080_gb300 import xlb as X

pytestmark = pytest.mark.gpu


def test_two_threads_step_lattices_of_different_sizes():
    shapes, errors, done = [(16, 33), (127, 126)], [], []

    def work(shape):
        try:
            s = X.Simulation(9, (shape[1], shape[0]), 1.4, "bgk", "f32")
            s.init(np.ones(shape, np.float32), np.zeros((2,) + shape, np.float32))
            for k in range(4000):
                s.step(2)
                if k % 200 == 0:
                    s.synchronize()
            s.synchronize()
            done.append(s.macroscopic()[0])
            s.close()
        except X.XlbError as e:
            errors.append(str(e))

    t = [threading.Thread(target=work, args=(sh,)) for sh in shapes]
    for x in t:
        x.start()
    for x in t:
        x.join()
    assert not errors and len(done) == 2
    assert all(np.allclose(r, 1.0, atol=1e-6) for r in done)
