"""The FP64 tanh and reciprocal square root that the kernels run (evaluate_math.cuh), on the
device, against mpmath: over their ranges and at the edges of their branches.

tanh: 4 units in the last place (its steps round some six times, two of them in a
factor near one).  1/sqrt: 2 units (a third-order step from an FP32 estimate, whose error
is below 1e-19, then two roundings); outside FP32's range it is CUDA's."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2603_01234_gb300 import build

pytestmark = pytest.mark.gpu
mp = pytest.importorskip("mpmath")
torch = pytest.importorskip("torch")
EPS = 2.0 ** -52
mp.mp.prec = 120
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def math64(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("math64") / "libmath64.so")
    r = subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", os.path.join(HERE, "math64_kernels.cu"), "-o", out],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = C.CDLL(out)

    def run(which, x):
        d = torch.from_numpy(np.ascontiguousarray(x, np.float64)).cuda()
        y = torch.empty_like(d)
        torch.cuda.synchronize()
        assert lib.math64(which, d.numel(), C.c_void_p(d.data_ptr()), C.c_void_p(y.data_ptr())) == 0
        return y.cpu().numpy()

    return run


def around(*values):
    """Each value with its neighbours on either side."""
    v = np.array(values)
    return np.concatenate([np.nextafter(v, -np.inf), v, np.nextafter(v, np.inf)])


def test_tanh(math64):
    rng = np.random.default_rng(1)
    edges = np.arange(0, 64) * np.log(2) / 64  # where the table's index changes
    x = np.concatenate([rng.uniform(-19.99, 19.99, 3000), rng.uniform(-1, 1, 3000), 10.0 ** rng.uniform(-300, 0, 1000),
                        around(*edges[1:], 19.0, 20.0, 21.0, 300.0, 1e300, 2.0 ** -1022, 2.0 ** -54)])
    x = np.concatenate([x, -x])
    want = np.array([float(mp.tanh(mp.mpf(float(v)))) for v in x])
    got = math64(0, x)
    assert np.all(np.abs(got - want) <= 4 * EPS * np.abs(want))
    np.testing.assert_array_equal(got[: x.size // 2], -got[x.size // 2:])
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324])
    np.testing.assert_array_equal(math64(0, special), [0.0, 0.0, 1.0, -1.0, np.nan, 5e-324])


def test_rsqrt(math64):
    rng = np.random.default_rng(2)
    low, high = 2.0 ** -126, 2.0 ** 128  # FP32's normal range
    x = np.concatenate([10.0 ** rng.uniform(-6, 6, 4000), 2.0 ** rng.uniform(-126, 128, 2000),
                        2.0 ** rng.uniform(-1022, 1023, 1000),
                        around(low, 2 * low, high, high / 2, 1.0, 4.0, 2.0 ** -149, 2.0 ** -1022, 2.0 ** 1023)])
    want = np.array([float(1 / mp.sqrt(mp.mpf(float(v)))) for v in x])
    assert np.all(np.abs(math64(1, x) - want) <= 2 * EPS * want)
    special = np.array([0.0, np.inf, -1.0, -np.inf, np.nan, -1e-3])
    np.testing.assert_array_equal(math64(1, special), [np.inf, 0.0, np.nan, np.nan, np.nan, np.nan])
