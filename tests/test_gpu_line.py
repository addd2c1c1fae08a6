"""One-dimensional FP32 members, whose whole step is one launch.

Against the oracle: every row length with more and fewer than half of the modes
kept, a variable bottom, the wavemaker's pressure, a sponge, the classical and
the integrating-factor steps.  Tolerances: after two steps the FP32 bar of the
other parity tests (1e-5 relative L2).  V weighs the short waves of smooth fields
and is the worse conditioned the longer the row, so its bar is taken from the
oracle: the change of its V when the inputs are rounded once to FP32, times 20
(some 50 sequential roundings, each of that size and of random sign, sqrt(50) = 7,
and a factor of 3).

Against itself: a member of a long row runs on as many blocks as the batch
leaves SMs for, and the results are the same bits for every number of blocks.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def sbi():
    import __graft_entry__ as g
    g.build()
    from paper_2310_19840_gb300 import sbi as s
    return s


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def single(a):
    return a.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("integrator", ["rk4", "lawson"])
@pytest.mark.parametrize("alpha", [0.34, 0.5, 1.0])
@pytest.mark.parametrize("nx", [16, 64, 128, 512, 1024, 2048, 4096])
def test_row_lengths_match_oracle(sbi, nx, alpha, integrator):
    from oracle import sbi_oracle as O
    L = 0.1 * nx
    grid = O.Grid(nx, 1, L)
    amp, omega, phase, x0 = [0.002, 0.001], [3.0, 5.5], [0.2, 1.1], 0.3 * L
    delta = W.random_field(nx, 1, 5, amplitude=0.02)
    sponge = W.random_field(nx, 1, 6, amplitude=1.0) ** 2
    pb = O.Problem(grid, 9.81, 0.7, delta=delta, alpha=alpha, order=4, sponge_w=sponge, sponge_nu=0.3,
                   wavemaker=O.Wavemaker(np.array(amp), np.array(omega), np.array(phase), x0), integrator=integrator)
    eta = O.project(pb, W.random_field(nx, 1, 7, amplitude=0.004, band=0.3))
    phi = O.project(pb, W.random_field(nx, 1, 8, amplitude=0.02, band=0.3))
    ctx = sbi.Context([(nx, 1, L, 1.0)], 9.81, [0.7 - delta], h0=0.7, order=4, alias_frac=alpha, sponge_w=sponge,
                      sponge_nu=0.3, integrator=sbi.SBI_LAWSON_RK4 if integrator == "lawson" else sbi.SBI_RK4)
    ctx.set_wavemaker(amp, omega, phase, x0)
    ctx.set_state(0, eta, phi)
    Vo = O.diagnose(pb, eta, phi)
    once = O.Problem(grid, 9.81, 0.7, delta=single(delta), alpha=alpha, order=4)
    assert rel(ctx.vertical_velocity(0), Vo) < 20 * rel(O.diagnose(once, single(eta), single(phi)), Vo)
    ctx.step(0.005, 2)
    e, p = ctx.get_state(0)
    eo, po = O.step(pb, eta, phi, 0.005, 2)
    assert rel(e, eo) < TOL and rel(p, po) < TOL
    ctx.close()


@pytest.mark.parametrize("nx, counts", [(256, (1, 5)), (2048, (1, 33, 65)), (4096, (1, 17, 33, 129))])
def test_a_member_alone_equals_it_in_a_batch(sbi, nx, counts):
    n = max(counts)
    eta = np.concatenate([W.random_field(nx, 1, 100 + i, amplitude=0.01).ravel() for i in range(n)])
    phi = np.concatenate([W.random_field(nx, 1, 200 + i, amplitude=0.05).ravel() for i in range(n)])
    out = {}
    for count in counts:
        ctx = sbi.Context([(nx, 1, 0.1 * nx, 1.0)] * count, 9.81, None, h0=0.7, filt_beta1=8.0, filt_beta2=30.0,
                          k_ref=1.0)
        ctx.set_wavemaker([0.002], [3.0], [0.2], 0.3)
        ctx.set_state_all(eta[:count * nx], phi[:count * nx])
        ctx.step(0.005, 2)
        e, p = ctx.get_state_all()
        out[count] = e[:nx], p[:nx]
        ctx.close()
    for count in counts[1:]:
        assert np.array_equal(out[count][0], out[1][0]) and np.array_equal(out[count][1], out[1][1]), count
