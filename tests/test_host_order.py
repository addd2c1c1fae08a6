"""The library's host code on a CUDA runtime that only keeps books (fake_cudart.cpp):
a stream's copies and fills happen when that stream is synchronised, no kernel
runs.  What a call leaves to chance on a GPU is then certain to go wrong here.
"""
import ctypes as C
import glob
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def built(tmp_path_factory):
    cxx, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not cxx or not os.path.exists(nvcc):
        pytest.skip("no compiler")
    import __graft_entry__ as g
    from paper_2310_19840_gb300 import build as b
    g.build()
    objs = [os.path.join(b.BUILD, os.path.splitext(s)[0] + ".o") for s in b.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        b.build(force=True)
    out = str(tmp_path_factory.mktemp("fake") / "libsbi_host.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", cuda,
                    os.path.join(ROOT, "tests", "fake_cudart.cpp"), *objs, "-Wl,-Bsymbolic", "-o", out], check=True)
    return out


@pytest.fixture
def host(built, monkeypatch):
    from paper_2310_19840_gb300 import sbi
    lib = C.CDLL(built)
    for name, (res, args) in sbi.EXPORTS.items():
        f = getattr(lib, name)
        f.restype, f.argtypes = res, args
    lib.fake_made_at.restype, lib.fake_made_at.argtypes = C.c_void_p, [C.c_int, C.POINTER(C.c_size_t)]
    lib.fake_live_bytes.restype = C.c_size_t
    monkeypatch.setattr(sbi, "_lib", lib)
    sbi.fake = lib
    yield sbi
    del sbi.fake


def doubles(lib, since):
    """The device allocations made from number `since` on, as float64 arrays."""
    out, n = [], C.c_size_t()
    for i in range(since, lib.fake_made()):
        p = lib.fake_made_at(i, C.byref(n))
        out.append(np.ctypeslib.as_array(C.cast(p, C.POINTER(C.c_double)), (n.value // 8,)).copy())
    return out


def test_time_and_wavemaker_outlast_the_zeroing_of_their_buffers(host):
    ctx = host.Context([(64, 1, 6.4, 1.0)], 9.81, None, h0=0.7)
    before = host.fake.fake_made()
    ctx.set_time(2.5)
    ctx.set_wavemaker([0.01, 0.02], [3.0, 4.0], [0.1, 0.2], 0.3)
    host.fake.fake_drain()
    time, params, profiles = doubles(host.fake, before)[:3]
    assert time[0] == 2.5
    assert list(params) == [3.0, 4.0, 0.1, 0.2]
    assert profiles.size == 128 and profiles.reshape(2, 64).max(axis=1).min() > 0
    ctx.close()


def test_streamed_passes_wait_for_their_tables(host):
    # a filtered step needs the table of Lambda only, the entry of the streamed
    # call the one of the mask
    grids = [(32, 16, 3.2, 1.6), (64, 32, 6.4, 3.2)]
    n = sum(g[0] * g[1] for g in grids)
    ctx = host.Context(grids, 9.81, None, h0=0.7, filt_beta1=8.0, filt_beta2=30.0, k_ref=1.0, autotune=0)
    a = np.zeros(n)
    ctx.step(0.01, 1)
    before = host.fake.fake_overtaken()
    ctx.step_streamed(a, a, 0.01, 1)
    assert host.fake.fake_overtaken() == before
    ctx.close()


@pytest.mark.parametrize("integrator", [0, 1, 2])
@pytest.mark.parametrize("diagnostic, bar, adapt", [(0, 0, 0.0), (0, 1, 0.0), (1, 0, 0.0), (0, 0, 1e-6), (0, 1, 1e-6)])
def test_a_one_dimensional_step_is_one_launch_between_adaptive_tests(host, integrator, diagnostic, bar, adapt):
    # at the highest order and with every term: the longest programs there are
    if integrator and adapt:
        pytest.skip("refused: the integrating factor takes no adapt_tol")
    nx = 64
    depth = np.full(nx, 0.7) - 0.1 * np.cos(2 * np.pi * np.arange(nx) / nx)
    ctx = host.Context([(nx, 1, 6.4, 1.0)], 9.81, [depth] if bar else None, h0=0.7, order=7, integrator=integrator,
                       diagnostic=diagnostic, adapt_tol=adapt, sponge_w=np.ones(nx), sponge_nu=0.3, filt_beta1=8.0,
                       filt_beta2=30.0, autotune=0)
    if integrator < 2:
        ctx.set_wavemaker([0.1] * 256, [1.0] * 256, [0.0] * 256, 0.0)
        ctx.step(0.01, 1)
        assert host.fake.fake_captured() == ctx.step_launches()
        assert adapt or ctx.step_launches() == 2       # with the time advance
    else:
        ctx.step_adaptive(0.001, 1e-3, 0.001)
    ctx.close()


@pytest.mark.parametrize("schemes", ["rk4", "wavemaker"])
def test_step_sizes_and_wavemakers_leave_no_programs_behind(host, schemes):
    # a program does not hold the step size; of those of earlier wavemakers at
    # most 32, and the one in use, are kept (40 KB each)
    nx = 64
    ctx = host.Context([(nx, 1, 6.4, 1.0)], 9.81, None, h0=0.7, autotune=0)
    ctx.set_wavemaker([0.1] * 256, [1.0] * 256, [0.0] * 256, 0.0)
    ctx.step(0.01, 1)
    held, made = host.fake.fake_live_bytes(), host.fake.fake_made()
    for k in range(100):
        if schemes == "rk4":
            ctx.step(0.01 + 1e-4 * (k + 1), 1)
        else:
            n = 1 + k
            ctx.set_wavemaker([0.1] * n, [1.0] * n, [0.0] * n, 0.0)
            ctx.step(0.01, 1)
    if schemes == "rk4":
        assert host.fake.fake_made() == made
    else:
        assert host.fake.fake_live_bytes() < held + 34 * 40960
    ctx.close()
    assert host.fake.fake_live_bytes() == 0


def test_the_wide_default_of_a_column_pass_is_among_the_timed_shapes(host):
    # the report gives chosen/default and the time of the chosen one (-1: none was
    # timed); at most one power of two more copies than transforms to share out
    import re
    ctx = host.Context([(64, 64, 6.4, 6.4)], 9.81, None, h0=0.7, order=4)
    ctx.step(0.01, 1)
    seen = set()
    for line in ctx.autotune_report().splitlines():
        m = re.match(r"col .* in=(\d+) .* out=(\d+) .*: cpb \S+/\S+w(\d+) (\S+) ms", line)
        if m:
            share = max(2, int(m[1]), int(m[2]))
            assert int(m[3]) < 2 * share and float(m[4]) > 0.0, line
            seen.add(share)
    assert 2 in seen and max(seen) > 2
    ctx.close()


@pytest.mark.parametrize("eights, size", [(16, 8), (15, 4)])
def test_clusters_of_a_batch_run_at_once(host, eights, size):
    host.fake.fake_max_clusters(8, eights)
    ctx = host.Context([(4096, 1, 409.6, 1.0)] * 16, 9.81, None, h0=0.7, order=3, autotune=0)
    ctx.step(0.01, 1)
    assert host.fake.fake_cluster_size() == size
    ctx.close()
