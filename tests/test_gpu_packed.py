"""The packed kernels of two-dimensional FP32 groups where they can go wrong.

Against the oracle: kept widths that leave the fast row form (more and fewer
than half of the modes, a count that is no multiple of four), every threads-per-
row and threads-per-column layout, several members, a sponge on a
two-dimensional grid, a flat and a variable bottom.  Tolerance: the FP32 bar of
the other parity tests (1e-5 relative L2 after one evaluation or two steps:
about 50 sequential roundings over the transforms, ~1e-6, times the conditioning
of the highest orders); the slopes are kept small enough that the wider masks
stay well conditioned.

Against itself: the forms that the launchers choose by size (products split over
blocks, wide column passes, rows and columns per block) give the same bits, so a
member alone equals the same member in a large batch.
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


@pytest.mark.parametrize("alpha", [0.34, 0.5, 0.8, 1.0])
@pytest.mark.parametrize("nx, ny", [(16, 8), (32, 32), (64, 128), (128, 16), (256, 64), (512, 8), (1024, 16), (2048, 8),
                                    (16, 256), (32, 512), (16, 1024), (16, 2048)])
def test_kept_widths_match_oracle(sbi, nx, ny, alpha):
    from oracle import sbi_oracle as O
    grid = O.Grid(nx, ny, 0.1 * nx, 0.1 * ny)
    variable = ny <= 32
    delta = W.random_field(nx, ny, 5, amplitude=0.02) if variable else None
    pb = O.Problem(grid, 9.81, 0.7, delta=delta, alpha=alpha, order=4,
                   sponge_w=W.random_field(nx, ny, 6, amplitude=1.0) ** 2, sponge_nu=0.3)
    eta = O.project(pb, W.random_field(nx, ny, 7, amplitude=0.004, band=0.3))
    phi = O.project(pb, W.random_field(nx, ny, 8, amplitude=0.02, band=0.3))
    ctx = sbi.Context([(nx, ny, 0.1 * nx, 0.1 * ny)], 9.81, [0.7 - delta if variable else None], h0=0.7, order=4,
                      alias_frac=alpha, sponge_w=pb.sponge_w, sponge_nu=0.3)
    ctx.set_state(0, eta, phi)
    V = ctx.vertical_velocity(0)
    Vo = O.diagnose(pb, eta, phi)
    assert rel(V, Vo) < TOL
    w = ctx.vertical_velocity(0, eulerian_w=True)
    ex, ey, _ = O.wavenumbers(grid)
    F = np.fft.fft2
    m = O.dealias_mask(grid, alpha)
    grad = lambda f: [np.real(np.fft.ifft2(1j * k * m * F(f))) for k in (ex, ey)]
    ge, gp = grad(eta), grad(phi)
    assert rel(w, (Vo + ge[0] * gp[0] + ge[1] * gp[1]) / (1 + ge[0] ** 2 + ge[1] ** 2)) < TOL
    ctx.step(0.005, 2)
    e, p = ctx.get_state(0)
    eo, po = O.step(pb, eta, phi, 0.005, 2)
    assert rel(e, eo) < TOL and rel(p, po) < TOL
    ctx.close()


@pytest.mark.parametrize("nx, ny, n", [(64, 64, 40), (256, 32, 33), (512, 128, 7), (128, 512, 9), (1024, 64, 3)])
def test_a_member_alone_equals_it_in_a_batch(sbi, nx, ny, n):
    # alone, a pass is split over blocks and its columns take the wide form; in
    # the batch (tuned and untuned) they do not
    spec = (nx, ny, 0.1 * nx, 0.1 * ny)
    eta = np.concatenate([W.random_field(nx, ny, 100 + i, amplitude=0.01).ravel() for i in range(n)])
    phi = np.concatenate([W.random_field(nx, ny, 200 + i, amplitude=0.05).ravel() for i in range(n)])
    out = {}
    for count, tune in ((1, 0), (n, 0), (n, 1)):
        ctx = sbi.Context([spec] * count, 9.81, None, h0=0.7, autotune=tune, filt_beta1=8.0, filt_beta2=30.0, k_ref=1.0)
        k = count * nx * ny
        ctx.set_state_all(eta[:k], phi[:k])
        ctx.step(0.005, 2)
        e, p = ctx.get_state_all()
        out[count, tune] = e[:nx * ny], p[:nx * ny]
        ctx.close()
    for key in ((n, 0), (n, 1)):
        assert np.array_equal(out[key][0], out[1, 0][0]) and np.array_equal(out[key][1], out[1, 0][1]), key


@pytest.mark.parametrize("alpha", [1.0 / 3.0, 0.75])
@pytest.mark.parametrize("nx, ny, n", [(64, 32, 70), (256, 128, 33), (512, 512, 6), (64, 1024, 12)])
def test_other_widths_alone_equal_the_batch(sbi, nx, ny, n, alpha):
    # the same for more and fewer than half of the modes: the wide column form of
    # every mode of a column, the rows' general form
    spec = (nx, ny, 0.1 * nx, 0.1 * ny)
    eta = np.concatenate([W.random_field(nx, ny, 100 + i, amplitude=0.004).ravel() for i in range(n)])
    phi = np.concatenate([W.random_field(nx, ny, 200 + i, amplitude=0.02).ravel() for i in range(n)])
    out = {}
    for count, tune in ((1, 0), (n, 0), (n, 1)):
        ctx = sbi.Context([spec] * count, 9.81, None, h0=0.7, order=4, alias_frac=alpha, autotune=tune)
        k = count * nx * ny
        ctx.set_state_all(eta[:k], phi[:k])
        ctx.step(0.005, 2)
        e, p = ctx.get_state_all()
        out[count, tune] = e[:nx * ny], p[:nx * ny]
        ctx.close()
    for key in ((n, 0), (n, 1)):
        assert np.array_equal(out[key][0], out[1, 0][0]) and np.array_equal(out[key][1], out[1, 0][1]), key
