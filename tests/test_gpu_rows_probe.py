"""Single device functions of the packed rows against what they stand for: the
quotient of the dynamic condition against IEEE division, bit for bit."""
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
