"""The reciprocal and the reflector that the spectral kernels build from hardware estimates, against division and square
roots over the exponents they may meet, and where the estimates give up (subnormal numbers)."""
import ctypes
import os
import subprocess
from pathlib import Path

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

HERE = Path(__file__).resolve().parent
CSRC = HERE.parent / "paper_2605_02905_b200" / "csrc"


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    so = tmp_path_factory.mktemp("fp64") / "fp64_probe.so"
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-shared",
                           "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "-I", str(CSRC), "-o", str(so), str(HERE / "fp64_probe.cu")])
    return ctypes.CDLL(str(so))


def _run(fn, *arrays, outputs):
    n = len(arrays[0])
    ins = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in arrays]
    outs = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(outputs)]
    torch.cuda.synchronize()
    assert fn(*[ctypes.c_void_p(t.data_ptr()) for t in ins + outs], n) == 0
    return [o.cpu().numpy() for o in outs]


def test_reciprocal(probe):
    """The third term of the series leaves 2^-60; the last multiply-add rounds by half a unit of 2^-52, the rest is held to another."""
    rng = np.random.default_rng(1)
    x = rng.choice([-1.0, 1.0], 200000) * rng.uniform(1.0, 2.0, 200000) * 2.0 ** rng.integers(-1000, 1000, 200000)
    y, = _run(probe.probe_rcp, x, outputs=1)
    assert np.max(np.abs(y / (1.0 / x) - 1.0)) < 4.5e-16


def test_reflector(probe):
    """beta and g within a few roundings of the exact ones, H orthogonal (u . u = 2), for |x| from 1e-140 to 1e140 and any
    share of it in the first entry."""
    rng = np.random.default_rng(2)
    n = 200000
    scale = 10.0 ** rng.uniform(-140, 140, n)
    alpha = rng.choice([-1.0, 1.0], n) * scale * 10.0 ** rng.uniform(-12, 0, n)
    rest = scale * 10.0 ** rng.uniform(-12, 0, n)
    alpha[:1000] = 0.0
    ss = rest * rest
    beta, g, amb = _run(probe.probe_reflector, alpha, ss, outputs=3)
    L = np.longdouble
    exact = np.sqrt(L(alpha) ** 2 + L(ss))
    want_beta = np.where(np.signbit(alpha), exact, -exact)
    want_g = 1.0 / np.sqrt(exact * (exact + np.abs(L(alpha))))
    assert float(np.max(np.abs(beta / want_beta - 1.0))) < 1e-15
    assert float(np.max(np.abs(g / want_g - 1.0))) < 1e-15
    assert np.array_equal(amb, alpha - beta)
    assert float(np.max(np.abs((L(amb) * g) ** 2 + L(ss) * L(g) ** 2 - 2.0))) < 8e-15


def test_reflector_of_next_to_nothing(probe):
    """Nothing to annihilate, and sums of squares that are not normal numbers: H = I, and never a NaN."""
    alpha = np.array([0.0, 3.0, -2.0, 0.0, 0.0, 1e-160, -1e-162, 1e-150, 1e10])
    ss = np.array([0.0, 0.0, 0.0, 5e-324, 1e-310, 1e-320, 1e-308, 1e-320, 1e-320])
    beta, g, amb = _run(probe.probe_reflector, alpha, ss, outputs=3)
    assert np.isfinite(beta).all() and np.isfinite(g).all() and np.isfinite(amb).all()
    assert np.array_equal(beta[:7], alpha[:7]) and not g[:7].any() and not amb[:7].any()
    np.testing.assert_allclose(beta[7:], -alpha[7:], rtol=1e-15)   # normal: the ordinary reflector
