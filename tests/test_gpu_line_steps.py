"""One-dimensional FP32 members whose step size changes from call to call: the
launch brings the step size, the program on the device stays.  Against the
oracle, with the tolerance of the other parity tests (1e-5 relative L2 after a
few steps)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("integrator", ["rk4", "lawson"])
@pytest.mark.parametrize("nx", [64, 2048])
def test_changing_step_sizes_match_oracle(nx, integrator):
    import __graft_entry__ as g
    g.build()
    from oracle import sbi_oracle as O
    from paper_2310_19840_gb300 import sbi
    L = 0.1 * nx
    grid = O.Grid(nx, 1, L)
    amp, omega, phase, x0 = [0.002, 0.001], [3.0, 5.5], [0.2, 1.1], 0.3 * L
    pb = O.Problem(grid, 9.81, 0.7, order=4, wavemaker=O.Wavemaker(np.array(amp), np.array(omega), np.array(phase), x0),
                   integrator=integrator)
    eta = O.project(pb, W.random_field(nx, 1, 7, amplitude=0.004, band=0.3))
    phi = O.project(pb, W.random_field(nx, 1, 8, amplitude=0.02, band=0.3))
    ctx = sbi.Context([(nx, 1, L, 1.0)], 9.81, None, h0=0.7, order=4,
                      integrator=sbi.SBI_LAWSON_RK4 if integrator == "lawson" else sbi.SBI_RK4)
    ctx.set_wavemaker(amp, omega, phase, x0)
    ctx.set_state(0, eta, phi)
    t, e, p = 0.0, eta, phi
    for dt in (0.005, 0.002, 0.007, 0.005):
        ctx.step(dt, 1)
        e, p = O.step(pb, e, p, dt, 1, t)
        t += dt
    got_e, got_p = ctx.get_state(0)
    assert np.linalg.norm(got_e - e) < 1e-5 * np.linalg.norm(e)
    assert np.linalg.norm(got_p - p) < 1e-5 * np.linalg.norm(p)
    ctx.close()
