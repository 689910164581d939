"""Synchronising calls of several threads on one context: each returns what it
asked for (more threads than the context has pinned slots from the start)."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_conservation_of_different_boxes_from_several_threads():
    from paper_0809_4958_gb300 import lbtracer as lbt
    lbt.load()
    sizes = [8, 16, 24, 32, 40, 48]
    tr = lbt.Tracers([lbt.box_desc(E, 0.8, periodic=(True, True, True)) for E in sizes], 0)
    for b, E in enumerate(sizes):
        tr.lb_init(b, np.full((3, E, E, E), 0.01 * (b + 1)))
    want = [list(tr.lb_conservation(b)) for b in range(len(sizes))]
    wrong = []

    def read(b):
        for _ in range(200):
            got = list(tr.lb_conservation(b))
            if got != want[b]:
                wrong.append((b, got))

    threads = [threading.Thread(target=read, args=(b,)) for b in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong[:3]
    for b, E in enumerate(sizes):
        assert abs(want[b][0] - E ** 3) < 1e-9 * E ** 3
    tr.close()
