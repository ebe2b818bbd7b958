"""Results at other addresses from call to call: totals into the places of an array in turn
(captured graphs replayed), at an address that is no multiple of eight bytes, in page-locked
memory, and device memory among the arrays of a host call on both sides of the size up to
which the CPU fills them.  Every value equals that of a call on arrays of its own."""
import ctypes as C

import numpy as np
import pytest

from paper_2603_01234_gb300 import binding, inputs
from tests.gpu_common import water_model

pytestmark = pytest.mark.gpu


def call(name, m, s, types, pos, energy, virial, force):
    """energy, virial: addresses."""
    lib, ptr = binding.load(), binding._ptr
    out = (C.c_void_p(energy), C.c_void_p(virial), None, ptr(force), None)
    if name == "batch":  # the configuration as two requests of half the particles each
        n = np.array([s.n // 2, s.n // 2], np.int32)
        h, which = (C.c_void_p * 1)(m.h.value), np.zeros(2, np.int32)
        box, pbc = np.tile(s.box, 2), np.tile(np.asarray(s.pbc, np.int32), 2)
        rc = lib.nep_compute_batch(C.cast(h, C.c_void_p), 1, 2, ptr(n), ptr(which), ptr(box), ptr(pbc), ptr(types), ptr(pos),
                                   binding.NEP_DEVICE, None, *out)
    else:
        one = (m.h, s.n, ptr(types), ptr(pos), ptr(s.box), ptr(np.asarray(s.pbc, np.int32)))
        rc = lib.nep_compute_static(*one, None, *out) if name == "static" else \
            lib.nep_compute(*one, binding.NEP_DEVICE, None, *out)
    binding._check(rc, name)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("name,requests", [("compute", 1), ("batch", 2), ("static", 1)])
def test_totals_at_other_addresses(nep_lib, name, requests, precision):
    torch = pytest.importorskip("torch")
    m = binding.Model(water_model(), precision)
    s = inputs.water_box(1000, seed=41)
    types, pos = torch.from_numpy(s.types).cuda(), torch.from_numpy(s.pos).cuda()
    force = torch.zeros(3, s.n, dtype=torch.float64, device="cuda")
    e, w = (torch.zeros(k * requests, dtype=torch.float64, device="cuda") for k in (1, 9))
    call(name, m, s, types, pos, e.data_ptr(), w.data_ptr(), force)
    want_e, want_w = e.cpu().numpy(), w.cpu().numpy()
    assert np.all(want_e != 0)
    E = torch.zeros(6, 1 * requests, dtype=torch.float64, device="cuda")
    W = torch.zeros(6, 9 * requests, dtype=torch.float64, device="cuda")
    for k in range(18):
        E[k % 6], W[k % 6] = 0, 0
        torch.cuda.synchronize()
        call(name, m, s, types, pos, E[k % 6].data_ptr(), W[k % 6].data_ptr(), force)
        np.testing.assert_array_equal(E[k % 6].cpu().numpy(), want_e)
        np.testing.assert_array_equal(W[k % 6].cpu().numpy(), want_w)
    raw = torch.zeros(512, dtype=torch.uint8, device="cuda")  # an address that is no multiple of eight
    for k in range(3):
        raw.zero_()
        torch.cuda.synchronize()
        call(name, m, s, types, pos, raw.data_ptr() + 4, raw.data_ptr() + 124, force)
        got = raw.cpu().numpy().tobytes()
        assert got[4:4 + 8 * requests] == want_e.tobytes() and got[124:124 + 72 * requests] == want_w.tobytes()
    pin = torch.zeros(64, dtype=torch.float64).pin_memory()
    call(name, m, s, types, pos, pin.data_ptr(), pin.data_ptr() + 160, force)
    np.testing.assert_array_equal(pin.numpy()[:requests], want_e)
    np.testing.assert_array_equal(pin.numpy()[20:20 + 9 * requests], want_w)
    m.close()


@pytest.mark.parametrize("n", [300, 4500])
def test_host_calls_with_device_memory_among_their_arrays(nep_lib, n):
    torch = pytest.importorskip("torch")
    m = binding.Model(water_model(), "fp32")
    s = inputs.water_box(n, seed=42)
    want = m.compute(s)
    out = {k: torch.zeros(v, dtype=torch.float64, device="cuda")
           for k, v in (("force", (3, n)), ("virial", (9, n)), ("site_energy", (n,)))}
    binding.nep_compute(m.h, s.types, s.pos, s.box, s.pbc, **out)
    for k, v in out.items():
        np.testing.assert_array_equal(v.cpu().numpy(), want[k])
    force = np.zeros((3, n))
    binding.nep_compute(m.h, torch.from_numpy(s.types).cuda(), s.pos, s.box, s.pbc, force=force)
    np.testing.assert_array_equal(force, want["force"])
    m.close()
