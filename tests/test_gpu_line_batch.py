"""Large ensembles of one-dimensional FP32 members, which run as one launch per pass
over all of them: the first, a middle and the last member against the oracle, on
either side of the size at which the form changes.  A variable bottom, the
wavemaker's pressure, a sponge, every row length, more and fewer than half of the
modes kept; tolerance: the FP32 bar of the other parity tests (1e-5 relative L2
after two steps)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx, n, alpha, bar, integrator, state64", [
    (16, 700, 0.5, False, "rk4", 0), (64, 456, 0.5, False, "rk4", 0), (64, 457, 0.5, False, "lawson", 0),
    (256, 609, 0.5, True, "rk4", 0), (256, 608, 0.5, True, "rk4", 1), (256, 460, 0.34, False, "rk4", 1),
    (1024, 457, 1.0, False, "lawson", 0), (2048, 153, 0.5, False, "rk4", 0), (2048, 305, 0.8, True, "rk4", 0),
    (4096, 153, 0.5, False, "rk4", 0)])
def test_large_ensembles_match_oracle(nx, n, alpha, bar, integrator, state64):
    import __graft_entry__ as g
    g.build()
    from oracle import sbi_oracle as O
    from paper_2310_19840_gb300 import sbi
    L = 0.1 * nx
    amp, omega, phase, x0 = [0.002, 0.001], [3.0, 5.5], [0.2, 1.1], 0.3 * L
    sponge = W.random_field(nx, 1, 6, amplitude=1.0) ** 2
    delta = W.random_field(nx, 1, 5, amplitude=0.02) if bar else None
    pb = O.Problem(O.Grid(nx, 1, L), 9.81, 0.7, delta=delta, alpha=alpha, order=4, sponge_w=sponge, sponge_nu=0.3,
                   wavemaker=O.Wavemaker(np.array(amp), np.array(omega), np.array(phase), x0), integrator=integrator)
    looked = (0, n // 2, n - 1)
    eta = np.zeros((n, nx))
    phi = np.zeros((n, nx))
    for m in looked:
        eta[m] = O.project(pb, W.random_field(nx, 1, 7 + m, amplitude=0.004, band=0.3))
        phi[m] = O.project(pb, W.random_field(nx, 1, 9 + m, amplitude=0.02, band=0.3))
    ctx = sbi.Context([(nx, 1, L, 1.0)] * n, 9.81, [0.7 - delta] * n if bar else None, h0=0.7, order=4,
                      alias_frac=alpha, sponge_w=sponge, sponge_nu=0.3, state_fp64=state64,
                      integrator=sbi.SBI_LAWSON_RK4 if integrator == "lawson" else sbi.SBI_RK4)
    ctx.set_wavemaker(amp, omega, phase, x0)
    ctx.set_state_all(eta.ravel(), phi.ravel())
    ctx.step(0.005, 2)
    e, p = (f.reshape(n, nx) for f in ctx.get_state_all())
    for m in looked:
        eo, po = O.step(pb, eta[m], phi[m], 0.005, 2)
        assert np.linalg.norm(e[m] - eo.ravel()) < 1e-5 * np.linalg.norm(eo), m
        assert np.linalg.norm(p[m] - po.ravel()) < 1e-5 * np.linalg.norm(po), m
    ctx.close()
