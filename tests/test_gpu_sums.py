"""Conservation sums (lb_conservation) against exactly rounded sums (math.fsum)
of the populations read back: every storage format, boxes of less than one
chunk of sites, of one chunk and a remainder, and of many chunks."""
import math

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [8, 16, 24, 40])
@pytest.mark.parametrize("storage", [0, 1, 2, 3])
def test_sums_match_exact_sums(storage, E):
    from paper_0809_4958_gb300 import lbtracer as lbt
    lbt.load()
    tr = lbt.Tracers([lbt.box_desc(E, 0.8, periodic=(True, True, True))], storage)
    rng = np.random.default_rng(E)
    tr.lb_init(0, np.ascontiguousarray(0.05 * rng.standard_normal((3, E, E, E)) * 10.0 ** rng.uniform(-6, 0, (1, E, E, E)),
                                       tr.np_real))
    got = tr.lb_conservation(0)
    d = tr.deviations(0).astype(np.float64).reshape(19, -1)
    c, _ = oracle.lattice()
    ref = [E ** 3 + math.fsum(d.ravel())] + [math.fsum((c[:, a].astype(float)[:, None] * d).ravel()) for a in range(3)]
    # an FP64 sum of n terms, however ordered, lies within n 2^-53 sum |d| of the exact one; the last addition of E^3
    bound = d.size * 2.0 ** -53 * np.abs(d).sum()
    assert abs(got[0] - ref[0]) <= bound + E ** 3 * 2.0 ** -52
    for a in range(3):
        assert abs(got[1 + a] - ref[1 + a]) <= bound
        if storage != 0:  # 72 bits a thread, then FP64 over the threads: 32 sites and more to a term
            assert abs(got[1 + a] - ref[1 + a]) <= bound / 16
    tr.close()
