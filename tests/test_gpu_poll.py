"""Polling: lb_sync with a short timeout on a busy stream returns after about
that time, however often it is called (calls that leave work behind on the
stream would fill its queue, and then wait for a place in it)."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_polling_a_busy_stream_stays_short():
    from paper_0809_4958_gb300 import lbtracer as lbt
    lbt.load()
    E = 256
    tr = lbt.Tracers([lbt.box_desc(E, 0.8, periodic=(True, True, True))], lbt.LB_STORE_F32)
    u0 = np.zeros((3, E, E, E), np.float32)
    u0[0] = 0.01
    tr.lb_init(0, u0)
    tr.lb_graph_capture(200)
    tr.lb_sync()
    t0 = time.monotonic()
    tr.lb_graph_launch()
    tr.lb_sync()
    one = time.monotonic() - t0
    for _ in range(int(5.0 / one) + 1):  # some five seconds of steps
        tr.lb_graph_launch()
    longest, polls, done = 0.0, 0, False
    while not done:
        t0 = time.monotonic()
        try:
            tr.lb_sync(0)
            done = True
        except lbt.LBError as e:
            assert e.code == lbt.LB_ERR_TIMEOUT
        longest = max(longest, time.monotonic() - t0)
        polls += 1
    print("%d polls, the longest %.1f ms" % (polls, 1e3 * longest))
    assert polls > 1500
    assert longest < 0.1  # a call waits one millisecond; the rest is the host's scheduling
    tr.close()
