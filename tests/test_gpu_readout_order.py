"""Read-outs enqueued right behind steps, without a synchronisation between:
density and velocity are those of the finished step, that is, bit for bit what
the same read-outs give once the stream has been waited for.  With and without
a chain (the kernel in front is the forced re-collision or the stream-collide
itself), on a box large enough that the read-out is resident before the step
has stored its last tiles."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nbeads", [0, 16])
@pytest.mark.parametrize("storage,E", [(0, 64), (1, 128), (2, 128), (3, 64)])
def test_fields_follow_the_step_before_them(storage, E, nbeads):
    import torch

    from paper_0809_4958_gb300 import inputs, lbtracer as lbt
    lbt.load()
    periodic = (nbeads == 0,) * 3
    tr = lbt.Tracers([lbt.box_desc(E, 0.7, periodic=periodic, nbeads=nbeads)], storage)
    rng = np.random.default_rng(3)
    tr.lb_init(0, np.ascontiguousarray(0.05 * rng.standard_normal((3, E, E, E)), tr.np_real))
    if nbeads:
        tr.chain_couple(0, lbt.chain_desc(nbeads), inputs.chain_start(1, nbeads, E))
        face = torch.zeros(18 * E * E, dtype=tr.real, device="cuda")
        torch.cuda.synchronize()
    pushed = -1
    rho = [torch.empty(E ** 3, dtype=tr.real, device="cuda") for _ in range(2)]
    u = [torch.empty(3 * E ** 3, dtype=tr.real, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    for n in range(12):
        while nbeads and pushed < n + 2:
            pushed += 1
            tr.lb_set_boundary(0, pushed, face)
        tr.lb_step(1)
        tr.lb_read_fields(0, lbt.LB_FIELD_RHO | lbt.LB_FIELD_ASYNC, rho[0])
        tr.lb_read_fields(0, lbt.LB_FIELD_U | lbt.LB_FIELD_ASYNC, u[0])
        tr.lb_sync()
        tr.lb_read_fields(0, lbt.LB_FIELD_RHO, rho[1])
        tr.lb_read_fields(0, lbt.LB_FIELD_U, u[1])
        assert torch.equal(rho[0], rho[1]) and torch.equal(u[0], u[1]), n
    tr.close()
