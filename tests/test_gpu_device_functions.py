"""The library's double-precision building blocks on the device, against the correctly rounded or extended-precision
values on the host."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1302_2132_gb300", "csrc")
SO = os.path.join(HERE, "_build", "libdevice_functions.so")


@pytest.fixture(scope="module")
def lib():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = os.path.join(HERE, "device_functions.cu")
    deps = [src] + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    os.makedirs(os.path.dirname(SO), exist_ok=True)
    if not os.path.exists(SO) or os.path.getmtime(SO) < max(os.path.getmtime(f) for f in deps):
        subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O3",
                               "-Xcompiler", "-fPIC", "-shared", "-I", CSRC, "-I",
                               os.path.join(os.path.dirname(os.path.dirname(CSRC)), "include"), "-o", SO + ".tmp", src])
        os.replace(SO + ".tmp", SO)
    return ctypes.CDLL(SO)


def apply(f, outputs, *args):
    """f(n, args..., outputs...) on device copies; args of n rows each."""
    n = len(args[0])
    dev = [torch.tensor(np.ascontiguousarray(a), device="cuda") for a in args]
    out = [torch.empty(n, dtype=t, device="cuda") for t in outputs]
    torch.cuda.synchronize()
    assert f(ctypes.c_long(n), *(ctypes.c_void_p(t.data_ptr()) for t in dev + out)) == 0
    return [t.cpu().numpy() for t in out]


def test_quotients_round_as_the_division_does(lib):
    rng = np.random.default_rng(4)
    n = 1 << 21
    a, b = (rng.uniform(1, 2, n) * 2.0 ** rng.integers(-40, 40, n) for _ in range(2))
    a *= rng.choice([-1.0, 1.0], n)
    b[:1000] = np.nextafter(2.0 ** rng.integers(-40, 40, 1000), 0)  # all ones in the significand
    (q,) = apply(lib.dev_quotient, [torch.float64], a, b)
    assert np.array_equal(q, a / b)


def test_double_states_near_zero_pressure(lib):
    """Physical if and only if the pressure that the oracle evaluates is positive: energies within two units in the
    last place of the kinetic energy."""
    rng = np.random.default_rng(8)
    n = 1 << 18
    rho, mu = rng.uniform(0.1, 4.0, n), rng.uniform(1.0, 50.0, n)
    kin = mu * mu / rho  # rounded as the oracle rounds it
    E = 0.5 * kin * (1 + rng.integers(-2, 3, n) * 2.0 ** -52)
    w = np.stack([rho, mu, np.zeros(n), E], 1)
    (ok,) = apply(lib.dev_physical, [torch.int32], w)
    assert np.array_equal(ok != 0, E > 0.5 * kin)


def test_reciprocal_square_root(lib):
    """No further from the exact value than 1 / sqrt(x) by two IEEE operations."""
    rng = np.random.default_rng(5)
    x = rng.uniform(1, 4, 1 << 20) * 4.0 ** rng.integers(-30, 30, 1 << 20)
    (y,) = apply(lib.dev_rsqrt, [torch.float64], x)
    exact = 1 / np.sqrt(x.astype(np.longdouble))
    ours, ieee = (np.abs((v - exact) / exact) for v in (y, 1 / np.sqrt(x)))
    assert ours.max() <= ieee.max() and np.mean(ours ** 2) <= np.mean(ieee ** 2)


def test_erfc_and_exponential(lib):
    """No further from the exact values than CUDA's own functions, in the largest and in the mean error, over the
    arguments whose erfc is a normal number; zero beyond."""
    rng = np.random.default_rng(6)
    x = np.concatenate([rng.uniform(-6, 26.5, 400000), rng.uniform(-3, 3, 400000), 10.0 ** rng.uniform(-12, 0, 50000)])
    c, e, cc, ce = apply(lib.dev_gauss, [torch.float64] * 4, x)
    assert np.array_equal(e, ce)
    hi, lo = np.empty_like(x), np.empty_like(x)
    ptr = lambda a: ctypes.c_void_p(a.ctypes.data)
    lib.host_erfc(ctypes.c_long(x.size), ptr(x), ptr(hi), ptr(lo))
    ours, theirs = (np.abs(((y - hi) - lo) / hi) for y in (c, cc))
    print("largest %.3g %.3g mean square root %.3g %.3g" % (ours.max(), theirs.max(), np.sqrt(np.mean(ours ** 2)),
                                                           np.sqrt(np.mean(theirs ** 2))))
    assert ours.max() <= theirs.max() and np.mean(ours ** 2) <= np.mean(theirs ** 2)
    c, e, _, _ = apply(lib.dev_gauss, [torch.float64] * 4, np.array([28.0, 40.0, 1e200, np.inf, -28.0, -np.inf, np.nan]))
    assert np.array_equal(c, [0, 0, 0, 0, 2, 2, np.nan], equal_nan=True) and not e[1:6].any() and np.isnan(e[6])
