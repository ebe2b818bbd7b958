"""The cell counters of a handle whose grids grow and shrink: a buffer that grows gets
more room than the grid at hand needs, and a later grid may use that room.  Every
result equals a fresh handle's."""
import numpy as np
import pytest

from paper_2603_01234_gb300 import binding, inputs
from tests.gpu_common import water_model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_grids_within_a_grown_buffer(nep_lib, precision):
    torch = pytest.importorskip("torch")
    model = water_model()
    m = binding.Model(model, precision)
    for nx in (10, 11, 12, 13, 9, 14):  # 100 ... 140 cells of 8 A; 110 grows the buffer to 125
        # what earlier allocations held is left in the memory that the library's next ones get
        junk = torch.full((1 << 22,), -1, dtype=torch.int32, device="cuda")
        del junk
        torch.cuda.empty_cache()
        box = np.array([8.0 * nx, 80.0, 8.0])
        rng = np.random.default_rng(nx)
        n = 400
        s = inputs.System(pos=np.ascontiguousarray(rng.uniform(0.0, 1.0, (3, n)) * box[:, None]),
                          types=np.zeros(n, np.int32), box=box, pbc=np.zeros(3, np.int32))
        got = m.compute(s)
        fresh = binding.Model(model, precision)
        want = fresh.compute(s)
        fresh.close()
        assert got["energy"] == want["energy"]
        np.testing.assert_array_equal(got["force"], want["force"])
        np.testing.assert_array_equal(got["virial"], want["virial"])
    m.close()


def test_fresh_handles_on_used_memory(nep_lib):
    """Handles created on memory that earlier ones filled and gave back, each taken through
    small grids of growing size: a buffer that is freed and allocated anew often comes back
    at the same address, with other contents behind its old end."""
    model = water_model()
    rng = np.random.default_rng(5)
    sizes = [64, 90, 130, 200, 300, 420, 150, 640, 800, 1000]
    systems = [inputs.water_box(n, seed=300 + n) for n in sizes]
    want = {}
    for rep in range(12):
        m = binding.Model(model, "fp32")
        for k in rng.permutation(len(systems)):
            got = m.compute(systems[k])
            ref = want.setdefault(int(k), got)
            assert got["energy"] == ref["energy"]
            np.testing.assert_array_equal(got["force"], ref["force"])
        m.close()
