"""The FP64 passes where they can go wrong: kept widths on both sides of half of
the modes (the column pass's register form and its general one), every column
and row length, several members, a sponge.  Tolerance: the FP64 bar of the other
parity tests (1e-10 relative L2).  A member alone equals the same member in a
batch, whose row passes run in fewer, longer blocks."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def sbi():
    import __graft_entry__ as g
    g.build()
    from paper_2310_19840_gb300 import sbi as s
    return s


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("alpha", [0.34, 0.5, 1.0])
@pytest.mark.parametrize("nx, ny", [(16, 8), (32, 16), (64, 32), (128, 64), (256, 128), (512, 256), (1024, 8), (2048, 8),
                                    (4096, 1), (16, 512), (16, 1024), (16, 2048)])
def test_kept_widths_match_oracle(sbi, nx, ny, alpha):
    from oracle import sbi_oracle as O
    grid = O.Grid(nx, ny, 0.1 * nx, 0.1 * ny)
    delta = W.random_field(nx, ny, 5, amplitude=0.02) if ny <= 64 else None
    pb = O.Problem(grid, 9.81, 0.7, delta=delta, alpha=alpha, order=4,
                   sponge_w=W.random_field(nx, ny, 6, amplitude=1.0) ** 2, sponge_nu=0.3)
    eta = O.project(pb, W.random_field(nx, ny, 7, amplitude=0.004, band=0.3))
    phi = O.project(pb, W.random_field(nx, ny, 8, amplitude=0.02, band=0.3))
    ctx = sbi.Context([(nx, ny, 0.1 * nx, 0.1 * ny)], 9.81, [None if delta is None else 0.7 - delta], h0=0.7, order=4,
                      precision=1, alias_frac=alpha, sponge_w=pb.sponge_w, sponge_nu=0.3)
    ctx.set_state(0, eta, phi)
    assert rel(ctx.vertical_velocity(0), O.diagnose(pb, eta, phi)) < TOL
    ctx.step(0.005, 2)
    e, p = ctx.get_state(0)
    eo, po = O.step(pb, eta, phi, 0.005, 2)
    assert rel(e, eo) < TOL and rel(p, po) < TOL
    ctx.close()


@pytest.mark.parametrize("nx, ny, n", [(64, 64, 40), (256, 32, 33), (512, 128, 7), (128, 512, 9)])
def test_a_member_alone_equals_it_in_a_batch(sbi, nx, ny, n):
    spec = (nx, ny, 0.1 * nx, 0.1 * ny)
    eta = np.concatenate([W.random_field(nx, ny, 100 + i, amplitude=0.01).ravel() for i in range(n)])
    phi = np.concatenate([W.random_field(nx, ny, 200 + i, amplitude=0.05).ravel() for i in range(n)])
    out = {}
    for count, tune in ((1, 0), (n, 0), (n, 1)):
        ctx = sbi.Context([spec] * count, 9.81, None, h0=0.7, precision=1, autotune=tune, filt_beta1=8.0,
                          filt_beta2=30.0, k_ref=1.0)
        k = count * nx * ny
        ctx.set_state_all(eta[:k], phi[:k])
        ctx.step(0.005, 2)
        e, p = ctx.get_state_all()
        out[count, tune] = e[:nx * ny], p[:nx * ny]
        ctx.close()
    for key in ((n, 0), (n, 1)):
        assert np.array_equal(out[key][0], out[1, 0][0]) and np.array_equal(out[key][1], out[1, 0][1]), key
