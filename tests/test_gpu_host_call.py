"""Host calls on either side of the size up to which the kernels work on page-locked memory
directly (4,096 particles) give the device call's bits, with all outputs and with only some
of them, and after a smaller and a larger call on the same handle."""
import numpy as np
import pytest

from paper_2603_01234_gb300 import binding, inputs
from tests.gpu_common import water_model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_host_calls_equal_device_calls(nep_lib, precision):
    torch = pytest.importorskip("torch")
    m = binding.Model(water_model(), precision)
    for n in (65, 4096, 4097, 130):
        s = inputs.water_box(n, seed=n)
        dev = m.compute_device(torch.from_numpy(s.types).cuda(), torch.from_numpy(s.pos).cuda(), s.box, s.pbc)
        host = m.compute(s)
        assert float(dev["energy"][0]) == host["energy"]
        for k in ("virial_total", "site_energy", "force", "virial"):
            np.testing.assert_array_equal(dev[k].cpu().numpy(), host[k])
        e, f = np.zeros(1), np.zeros((3, n))
        binding.nep_compute(m.h, s.types, s.pos, s.box, s.pbc, energy_total=e)  # totals alone
        assert e[0] == host["energy"]
        binding.nep_compute(m.h, s.types, s.pos, s.box, s.pbc, force=f)  # forces alone
        np.testing.assert_array_equal(f, host["force"])
    m.close()
