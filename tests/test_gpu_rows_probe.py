"""Single device functions of the packed rows against what they stand for: the
quotient of the dynamic condition against IEEE division, bit for bit; the factors
of a transform's third pass against their values, in units of 2^-24: powers up to
the seventh by at most three products of table entries.  An entry is off by 0.34
(root mean square), and forming the powers in correctly rounded operations gives
0.34, 0.87 and 0.89 for 512, 1024 and 2048 elements; the bounds are 1.1 times
that.  (Powers of a product in place of the entry: 0.63, 1.42 and 1.33.)"""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("probe") / "probe.so")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O3", "-Xcompiler", "-fPIC",
                    "-shared", "-I", os.path.join(ROOT, "paper_2310_19840_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "rows_probe.cu"), "-o", out], check=True)
    lib = C.CDLL(out)
    lib.probe_quotients.argtypes = [C.c_void_p] * 3 + [C.c_int]
    lib.probe_third_pass.argtypes = [C.c_int, C.c_void_p, C.c_void_p]
    return lib


def test_quotients_are_ieee_divisions(probe):
    import torch
    rng = np.random.default_rng(3)
    n = 1 << 18
    d = (2.0 ** rng.uniform(0, 127.9, n)).astype(np.float32)
    d[: n // 2] = (1.0 + 10.0 ** rng.uniform(-8, 1, n // 2)).astype(np.float32)
    a = (rng.standard_normal(n) * 2.0 ** rng.uniform(-40, 126, n)).astype(np.float32)
    a[: n // 2] = (rng.standard_normal(n // 2) * 10.0 ** rng.uniform(-6, 2, n // 2)).astype(np.float32)
    a[:8] = [0.0, 1.0, -1.0, np.inf, np.inf, np.nan, 3e38, 1e-30]
    d[:8] = [np.inf, np.inf, 3e38, 2.0, np.inf, 1.0, 3e38, 3e38]
    ta, td = torch.tensor(a).cuda(), torch.tensor(d).cuda()
    out = torch.empty_like(ta)
    assert probe.probe_quotients(ta.data_ptr(), td.data_ptr(), out.data_ptr(), n // 2) == 0
    with np.errstate(all="ignore"):
        want = a / d
    got = out.cpu().numpy()
    assert np.array_equal(got, want, equal_nan=True)


@pytest.mark.parametrize("n, bound", [(512, 0.38), (1024, 0.96), (2048, 0.98)])
def test_third_pass_factors(probe, n, bound):
    import torch
    table = np.zeros((8192 * 2 - 2, 2), np.float32)
    for N in [2 ** q for q in range(1, 14)]:
        a = -2.0 * np.pi * np.arange(N) / N
        table[N - 2:2 * N - 2] = np.stack([np.cos(a), np.sin(a)], 1)
    tw = torch.tensor(table).cuda()
    rp = n // 256
    out = torch.zeros((rp, n // rp, 2), dtype=torch.float32, device="cuda")
    assert probe.probe_third_pass(n, tw.data_ptr(), out.data_ptr()) == 0
    got = out.cpu().numpy().astype(np.float64)[1:]
    want = np.exp(-2j * np.pi * np.outer(np.arange(1, rp), np.arange(n // rp)) / n)
    err = np.abs(got[..., 0] + 1j * got[..., 1] - want)
    assert np.sqrt(np.mean(err ** 2)) < bound * 2.0 ** -24
