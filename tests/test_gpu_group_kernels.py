"""The evaluation kernels with a group of lanes per particle and those with a thread per
particle give the same bits: a configuration alone (few work items: group kernels)
equals itself inside a batch of more work items than those take, for every small parity
case in the FP32 and BF16 forms and with the four- and five-body terms.  And MD steps of
a system large enough for the thread-per-particle kernels, whose output pass applies the
closing kick, follow the FP64 form's."""
import numpy as np
import pytest

from paper_2603_01234_gb300 import binding, inputs
from tests.gpu_common import rms, small_systems, water_model

pytestmark = pytest.mark.gpu

GROUP_MAX_ITEMS = 200  # kGroupMaxItems of evaluate.cu


def cases():
    for name, model, system in small_systems():
        yield name, model, system
    for nr, na, k in ((5, 4, 8), (5, 5, 9)):
        m = inputs.random_model(n_types=2, n_desc_radial=nr, n_desc_angular=na, n_basis_radial=k, n_basis_angular=k,
                                hidden=35, rc_radial=6.0, rc_angular=4.5, seed=21, l_max_4b=2, l_max_5b=1)
        yield f"manybody{na}", m, inputs.random_periodic(300, [16.0, 17.0, 18.0], seed=22, min_dist=1.5, n_types=2)
    m = inputs.random_model(n_types=1, hidden=33, rc_radial=8.0, rc_angular=5.0, seed=23, l_max_4b=2)
    yield "fourbody_one_type", m, inputs.water_box(130, seed=24)


CASES = list(cases())


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("name,model,system", CASES, ids=[c[0] for c in CASES])
def test_group_and_thread_kernels_agree(nep_lib, name, model, system, precision):
    h = binding.Model(model, precision)
    alone = h.compute(system)
    copies = GROUP_MAX_ITEMS // -(-system.n // 128) + 1
    req_n, req_box, req_pbc, types, pos = binding.pack_requests([system] * copies)
    n = int(req_n.sum())
    e, wt, U, F, W = np.zeros(copies), np.zeros((copies, 9)), np.zeros(n), np.zeros(3 * n), np.zeros(9 * n)
    binding.nep_compute_batch([h.h], req_n, np.zeros(copies), req_box, req_pbc, types, pos, e, wt, U, F, W)
    Fs, Ws = binding.unpack_blocks(F, req_n, 3), binding.unpack_blocks(W, req_n, 9)
    for r in (0, copies - 1):
        np.testing.assert_array_equal(U[r * system.n:(r + 1) * system.n], alone["site_energy"])
        np.testing.assert_array_equal(Fs[r], alone["force"])
        np.testing.assert_array_equal(Ws[r], alone["virial"])
        np.testing.assert_array_equal(wt[r], alone["virial_total"])
        assert e[r] == alone["energy"]
    h.close()


def test_large_md_follows_fp64(nep_lib):
    """Two steps with a thermo row each: velocities differ by the FP32 force error only
    (forces within 1e-4 F_rms + 1e-6 of FP64's, the parity bound, at both ends of a step)."""
    s = inputs.water_box(27_000, seed=25)  # 211 work items
    s.masses = np.array([18.0])
    v = inputs.maxwell_boltzmann(s, 300.0, seed=26)
    got = {}
    for precision in ("fp32", "fp64"):
        m = binding.Model(water_model(), precision)
        pos, vel, force, th = s.pos.copy(), v.copy(), np.zeros_like(s.pos), np.zeros((2, 12))
        binding.nep_md_step(m.h, s.types, s.masses, s.box, s.pbc, pos, vel, force, 0, 2, 2.0, 1, th)
        got[precision] = (pos, vel, force, th)
        m.close()
    f_err = 1e-4 * rms(got["fp64"][2]) + 1e-6
    v_err = 2 * 2.0 * inputs.ACC_EV_A_AMU / 18.0 * f_err  # two steps of dt = 2 fs
    assert np.abs(got["fp32"][2] - got["fp64"][2]).max() <= f_err
    assert np.abs(got["fp32"][1] - got["fp64"][1]).max() <= v_err
    np.testing.assert_allclose(got["fp32"][3][:, 1:3], got["fp64"][3][:, 1:3], rtol=1e-5)
