"""The thread-per-particle kernels of the FP32 form, at sizes where no rule takes the group or
the warp kernels: every compiled variant gives the same bits, and so does a configuration
in a batch beyond the warp kernels' and alone (one warp per particle)."""
import numpy as np
import pytest

from paper_2603_01234_gb300 import binding, inputs
from tests.gpu_common import monolayer_model, small_systems, water_model

pytestmark = pytest.mark.gpu
PARTICLES = 70_000  # beyond every rule's line for the group and the warp kernels (dispatch.h)


@pytest.mark.parametrize("name", ["water", "monolayer"])
def test_variants_identical_and_autotune(nep_lib, name):
    """2 or 3 blocks per SM of the descriptor kernel; 3, 4 or 5 of the radial kernel with walk groups
    of 4 or 8 entries."""
    if name == "water":
        model, s = water_model(), inputs.water_box(27_001, seed=17)
    else:
        model, s = monolayer_model(), inputs.monolayer(83, 83, seed=18)
    m = binding.Model(model, "fp32")
    ref = None
    for md in (2, 3):
        for mf in (3, 4, 5):
            for ch in (4, 8):
                binding.nep_set_tuning(m.h, 0, md, mf, ch)
                got = m.compute(s)
                ref = ref or got
                assert got["energy"] == ref["energy"]
                for k in ("virial_total", "site_energy", "force", "virial"):
                    np.testing.assert_array_equal(got[k], ref[k])
    chosen = binding.nep_autotune(m.h, s.types, s.pos, s.box, s.pbc)
    assert chosen[0] in (2, 3) and chosen[1] in (3, 4, 5) and chosen[2] in (4, 8)
    got = m.compute(s)
    np.testing.assert_array_equal(got["force"], ref["force"])
    m.close()


@pytest.mark.parametrize("case", list(small_systems()), ids=[c[0] for c in small_systems()])
def test_small_systems_in_a_large_batch(nep_lib, case):
    """Tiny boxes whose stencils repeat cells as images, open axes, several types: alone and inside
    a batch of copies."""
    name, model, system = case
    h = binding.Model(model, "fp32")
    alone = h.compute(system)
    copies = PARTICLES // system.n + 1
    req_n, req_box, req_pbc, types, pos = binding.pack_requests([system] * copies)
    n = int(req_n.sum())
    e, wt, U, F, W = np.zeros(copies), np.zeros((copies, 9)), np.zeros(n), np.zeros(3 * n), np.zeros(9 * n)
    binding.nep_compute_batch([h.h], req_n, np.zeros(copies), req_box, req_pbc, types, pos, e, wt, U, F, W)
    Fs, Ws = binding.unpack_blocks(F, req_n, 3), binding.unpack_blocks(W, req_n, 9)
    for r in (0, copies // 2, copies - 1):
        np.testing.assert_array_equal(U[r * system.n:(r + 1) * system.n], alone["site_energy"])
        np.testing.assert_array_equal(Fs[r], alone["force"])
        np.testing.assert_array_equal(Ws[r], alone["virial"])
        np.testing.assert_array_equal(wt[r], alone["virial_total"])
        assert e[r] == alone["energy"]
    h.close()
