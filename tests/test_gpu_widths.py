"""Kept widths next to the borders between the forms of a packed row (half of the
modes, fewer, more): two modes, one below half, one above, all but one.  Against
the oracle, with the FP32 bar of the other parity tests (1e-5 relative L2)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kept", ["two", "half - 1", "half + 1", "all - 1"])
@pytest.mark.parametrize("nx, ny", [(16, 16), (32, 8), (64, 32), (512, 16), (1024, 8), (2048, 8), (16, 1024), (32, 2048)])
def test_widths_at_the_borders_match_oracle(nx, ny, kept):
    import __graft_entry__ as g
    g.build()
    from oracle import sbi_oracle as O
    from paper_2310_19840_gb300 import sbi
    n = nx // 2                              # modes of a row; W of them kept
    w = {"two": 2, "half - 1": n // 2 - 1, "half + 1": n // 2 + 1, "all - 1": n - 1}[kept]
    alpha = (w - 0.5) / n                    # kept: m < alpha n
    grid = O.Grid(nx, ny, 0.1 * nx, 0.1 * ny)
    pb = O.Problem(grid, 9.81, 0.7, alpha=alpha, order=3,
                   sponge_w=W.random_field(nx, ny, 6, amplitude=1.0) ** 2, sponge_nu=0.3)
    eta = O.project(pb, W.random_field(nx, ny, 7, amplitude=0.004, band=0.3))
    phi = O.project(pb, W.random_field(nx, ny, 8, amplitude=0.02, band=0.3))
    ctx = sbi.Context([(nx, ny, 0.1 * nx, 0.1 * ny)], 9.81, None, h0=0.7, order=3, alias_frac=alpha,
                      sponge_w=pb.sponge_w, sponge_nu=0.3)
    ctx.set_state(0, eta, phi)
    V, Vo = ctx.vertical_velocity(0), O.diagnose(pb, eta, phi)
    assert np.linalg.norm(V - Vo) < 1e-5 * np.linalg.norm(Vo)
    ctx.step(0.005, 2)
    e, p = ctx.get_state(0)
    eo, po = O.step(pb, eta, phi, 0.005, 2)
    assert np.linalg.norm(e - eo) < 1e-5 * np.linalg.norm(eo)
    assert np.linalg.norm(p - po) < 1e-5 * np.linalg.norm(po)
    ctx.close()
