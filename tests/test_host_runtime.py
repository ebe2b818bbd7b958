"""The library's host code (csrc/capi.cu) on the stand-in CUDA runtime of tests/host_runtime:
what it allocates, keeps and hands to the kernels, when an allocation fails or a buffer
moves.  Every array that a kernel would touch is checked against the live allocations."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2603_01234_gb300 import binding, inputs

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def host_library(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("host") / "libnep_host.so")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-fPIC", "-shared", "-Wl,-Bsymbolic",
                        "-I", os.path.join(HERE, "host_runtime"), "-I", os.path.join(os.path.dirname(HERE), "include"),
                        os.path.join(HERE, "host_runtime", "nep_host.cpp"), "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


class Host:
    def __init__(self, lib):
        self.lib = lib
        lib.host_counter.restype = C.c_long
        lib.host_set.argtypes = [C.c_char_p, C.c_long]
        lib.host_allocate.restype = C.c_void_p
        lib.host_allocate.argtypes = [C.c_int, C.c_size_t]
        lib.host_copies.restype = C.c_long
        lib.host_copies.argtypes = [C.c_void_p]
        for what, value in (("fail_in", -1), ("fail_host_in", -1), ("needR", 20), ("needA", 10)):
            self.set(what, value)
        lib.host_reset_counters()

    def set(self, what, value):
        self.lib.host_set(what.encode(), value)

    def count(self, what):
        return self.lib.host_counter(what.encode())

    def check(self):
        """No kernel was given an array that is not there, nor cell counters that are not zero."""
        assert self.count("bad") == 0 and self.count("uncleared") == 0


@pytest.fixture
def host(host_library, monkeypatch):
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "library_path", lambda: host_library)
    return Host(binding.load())


def model():
    return inputs.random_model(n_types=1, hidden=5, rc_radial=4.0, rc_angular=3.0, seed=1)


def system(n, box=(12.0, 12.0, 12.0)):
    rng = np.random.default_rng(n)
    return inputs.System(pos=np.ascontiguousarray(rng.uniform(0, 1, (3, n)) * np.array(box)[:, None]),
                         types=np.zeros(n, np.int32), box=np.array(box), pbc=np.ones(3, np.int32))


def with_failures(host, prepare, call):
    """Handles on which call() failed at its first, second, ... device allocation, until none is
    left to fail."""
    for k in range(200):
        h = prepare()
        host.set("fail_in", k)
        try:
            call(h)
            ended = True
        except binding.NepError as e:
            assert e.code == binding.NEP_ERR_OOM
            ended = False
        host.set("fail_in", -1)
        yield h
        host.check()
        h.close()
        if ended:
            return
    raise AssertionError("allocations without end")


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_lists_after_a_failed_allocation(host, precision):
    """A call that runs out of memory while it grows the neighbour lists or the pair forces
    leaves the handle usable: the size that worked before works again, and so does the call."""
    small, large = system(300), system(6000)

    def prepare():
        m = binding.Model(model(), precision)
        m.compute(small)
        return m

    for m in with_failures(host, prepare, lambda m: m.compute(large)):
        m.compute(small)
        m.compute(large)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_lists_after_a_failed_growth(host, precision):
    """The same when the lists grow because a configuration has more neighbours."""
    s = system(300)

    def prepare():
        host.set("needR", 20), host.set("needA", 10)
        m = binding.Model(model(), precision)
        m.compute(s)
        host.set("needR", 500), host.set("needA", 400)
        return m

    for m in with_failures(host, prepare, lambda m: m.neighbors(s, 0, 4)):
        m.compute(s)


@pytest.mark.parametrize("later", [(40.0, 40.0, 40.0), (28.0, 28.0, 28.0)])
def test_cell_counters_after_a_failed_allocation(host, later):
    """A call that runs out of memory while it grows the cell arrays leaves counters that the
    next build, of the same grid or of a smaller one, clears before it counts."""
    first, large, then = system(300), system(300, (40.0, 40.0, 40.0)), system(300, later)

    def prepare():
        m = binding.Model(model(), "fp32")
        m.compute(first)
        return m

    for m in with_failures(host, prepare, lambda m: m.compute(large)):
        m.compute(then)
        m.compute(large)


def batch(m, requests):
    req_n, box, pbc, types, pos = binding.pack_requests(requests)
    energy = np.zeros(len(requests))
    binding.nep_compute_batch([m.h], req_n, np.zeros(len(requests), np.int32), box, pbc, types, pos, energy)
    return energy


def test_plan_tables_after_a_failed_allocation(host):
    """A batch whose tables get a new device buffer but no staging for their upload leaves no
    plan that a later call would take for its own."""
    m = binding.Model(model(), "fp32")
    small, many = system(300), [system(2)] * 300
    m.compute(small)
    host.set("fail_host_in", 0)
    with pytest.raises(binding.NepError) as e:
        batch(m, many)
    assert e.value.code == binding.NEP_ERR_OOM
    assert m.compute(small)["energy"] == 0.5
    assert list(batch(m, many)) == [r + 0.5 for r in range(300)]
    host.check()
    m.close()


class DeviceCall:
    """nep_compute (or its variants) on arrays of the stand-in device, one configuration."""

    def __init__(self, host, m, s):
        self.m, self.s, self.host = m, s, host
        self.types, self.pos = self.device(s.types), self.device(s.pos)
        self.force = self.device(np.zeros((3, s.n)))

    def device(self, a):
        p = self.host.lib.host_allocate(2, a.nbytes)
        C.memmove(p, a.ctypes.data, a.nbytes)
        return p

    def __call__(self, name, energy, virial):
        lib, s, ptr = self.host.lib, self.s, binding._ptr
        one = (self.types, self.pos, ptr(s.box), ptr(s.pbc))
        out = (energy, virial, None, self.force, None)
        if name == "batch":  # two requests of the one configuration's halves
            n = np.array([s.n // 2, s.n - s.n // 2], np.int32)
            box, pbc = np.tile(s.box, 2), np.tile(s.pbc, 2)
            h, which = (C.c_void_p * 1)(self.m.h), np.zeros(2, np.int32)
            rc = lib.nep_compute_batch(C.cast(h, C.c_void_p), 1, 2, ptr(n), ptr(which), ptr(box), ptr(pbc), self.types,
                                       self.pos, binding.NEP_DEVICE, None, *out)
        elif name == "static":
            rc = lib.nep_compute_static(self.m.h, s.n, *one, None, *out)
        else:
            rc = lib.nep_compute(self.m.h, s.n, *one, binding.NEP_DEVICE, None, *out)
        binding._check(rc, name)


def doubles(address, count):
    return list(np.frombuffer(C.string_at(address, 8 * count)))


@pytest.mark.parametrize("name,requests", [("compute", 1), ("batch", 2), ("static", 1)])
def test_totals_at_other_addresses_replay_one_graph(host, name, requests):
    """A program that takes each frame's totals into another place, its other arrays staying
    where they are, replays one captured graph."""
    m = binding.Model(model(), "fp32")
    call = DeviceCall(host, m, system(300))
    E, W = call.device(np.zeros(2 * 40)), call.device(np.zeros(18 * 40))
    for k in range(200):
        at = k % 40
        e, w = E + 16 * at, W + 144 * at
        C.memset(e, 0, 8 * requests), C.memset(w, 0, 72 * requests)
        call(name, e, w)
        assert doubles(e, requests) == [0.5, 1.5][:requests]
        assert doubles(w, 9 * requests) == [float(r + c) for r in range(requests) for c in range(9)]
        if name != "static":  # launched once by itself and once into the graph
            assert host.count("evaluate") == min(k, 1) + 1 and host.count("instantiate") == min(k, 1)
    host.check()
    m.close()


@pytest.mark.parametrize("where", ["unaligned", "other_device", "page_locked"])
@pytest.mark.parametrize("name,requests", [("compute", 1), ("batch", 2), ("static", 1)])
def test_totals_where_the_kernels_cannot_write(host, name, requests, where):
    """Totals at an address that is no multiple of eight bytes, or on a device that the kernels do
    not reach, arrive by a copy; no kernel gets such an address."""
    m = binding.Model(model(), "fp32")
    call = DeviceCall(host, m, system(300))
    kind = {"unaligned": 2, "other_device": 3, "page_locked": 1}[where]
    e, w = (host.lib.host_allocate(kind, 1024) + (4 if where == "unaligned" else 0) for _ in range(2))
    for k in range(3):
        C.memset(e, 0, 8 * requests), C.memset(w, 0, 72 * requests)
        call(name, e, w)
        assert doubles(e, requests) == [0.5, 1.5][:requests]
        assert doubles(w, 9 * requests) == [float(r + c) for r in range(requests) for c in range(9)]
    host.check()
    m.close()


def test_small_host_calls_with_device_memory_among_their_arrays(host):
    """A small host call works on page-locked memory that the CPU fills and reads.  Device memory,
    which the CPU cannot reach, goes through copies, as in larger calls."""
    m = binding.Model(model(), "fp32")
    s, ptr = system(300), binding._ptr
    call = DeviceCall(host, m, s)
    host_force = np.zeros((3, s.n))
    for types, pos, force in ((call.types, ptr(s.pos), ptr(host_force)), (ptr(s.types), call.pos, ptr(host_force)),
                              (ptr(s.types), ptr(s.pos), call.force)):
        copied = {p: host.lib.host_copies(p) for p in (call.types, call.pos, call.force)}
        rc = host.lib.nep_compute(m.h, s.n, types, pos, ptr(s.box), ptr(s.pbc), binding.NEP_HOST, None, None, None, None,
                                  force, None)
        binding._check(rc, "nep_compute")
        for p in copied:
            assert (host.lib.host_copies(p) > copied[p]) == (p in (types, pos, force))
    host.check()
    m.close()


def test_small_host_calls_allocate_their_buffer_once(host):
    """Host calls of rising size keep one page-locked buffer, and a size seen twice before replays
    its graph after larger ones."""
    m = binding.Model(model(), "fp32")
    m.compute(system(4096))
    before = host.count("malloc_host")
    for n in (100, 200, 300, 400, 4096):
        m.compute(system(n))
    assert host.count("malloc_host") == before
    m.close()
    m = binding.Model(model(), "fp32")
    m.compute(system(100))
    before = host.count("malloc_host")
    for n in (200, 300, 400):
        m.compute(system(n))
    assert host.count("malloc_host") == before
    host.check()
    m.close()


def test_fp64_first_sizing_of_a_thin_open_box(host):
    """The first estimate of the list capacities from the box's density knows nothing of an open
    axis: a sheet in a flat box is estimated at the ceiling of 4,096.  With the FP64 form's pair
    forces (24 bytes an angular slot) that is no more memory than two lists of the ceiling and
    800 bytes a particle, and a configuration that needs more angular slots still gets them."""
    n = 2000
    s = system(n, (100.0, 100.0, 0.01))
    s.pbc[2] = 0
    m = binding.Model(model(), "fp64")
    asked = binding.nep_request_workspace([m.h], 0, n, s.box, s.pbc)
    m.compute(s)
    radial, angular = binding.nep_get_capacity(m.h)
    lists = 4 * (radial + angular) + 24 * angular
    assert radial == 4096 and lists <= 2 * 4 * 4096 + 800
    others = 600  # records, gradients, totals and staging of a particle: see nep_request_workspace
    assert binding.nep_workspace_bytes(m.h) <= asked <= n * (lists + others) + 100_000
    host.set("needA", 1000)
    m.compute(s)
    assert binding.nep_get_capacity(m.h)[1] >= 1000
    host.check()
    m.close()


def neighbor_form(host, boxes, fp64=False):
    """boxes: (particles, box, pbc, types, r_c) of each request."""
    arr = lambda k, t: np.ascontiguousarray([b[k] for b in boxes], t)  # noqa: E731
    n, box, pbc, types, rc = arr(0, np.int32), arr(1, np.float64), arr(2, np.int32), arr(3, np.int32), arr(4, np.float64)
    p = binding._ptr
    return host.lib.host_neighbor_form(len(boxes), p(n), p(types), p(box), p(pbc), p(rc), int(fp64))


def water(n, types=1):
    return n, [(n / 0.0334) ** (1 / 3)] * 3, [1, 1, 1], types, 8.0


def monolayer(n):
    s = inputs.monolayer(max(2, round((n / 4) ** 0.5)), max(2, round(n / 4 / max(2, round((n / 4) ** 0.5)))))
    return s.n, s.box, s.pbc, 4, 15.0


def test_neighbour_kernel_of_a_batch(host):
    """The kernel that measured fastest (or within a few percent of it) at sizes where the choice
    costs most."""
    for n, want in ((2_000, 1), (9_000, 1), (30_000, 8), (50_000, 0), (60_000, 0), (100_000, 0)):
        assert neighbor_form(host, [water(n)]) == want, n
    for n, want in ((9_000, 1), (30_000, 8), (58_000, 8), (77_000, 0)):
        assert neighbor_form(host, [water(n, types=2)]) == want, n
    assert neighbor_form(host, [monolayer(50_000)]) == 0 and neighbor_form(host, [monolayer(4_000)]) == 1
    wire = inputs.nanowire(60_001, n_cells_x=196)
    assert neighbor_form(host, [(wire.n, wire.box, wire.pbc, 3, 7.0)]) == 8
    # batches: what counts is the densest request's tests against everyone's
    assert neighbor_form(host, [water(100)] * 250) == 0 and neighbor_form(host, [water(100)] * 60) == 1
    rng = np.random.default_rng(7)
    sizes = np.exp(rng.uniform(np.log(64), np.log(1000), 100)).astype(int)
    assert neighbor_form(host, [water(n) if k % 2 else monolayer(n) for k, n in enumerate(sizes)]) == 1
    assert neighbor_form(host, [water(11_000)], fp64=True) == 1 and neighbor_form(host, [water(12_000)], fp64=True) == 0


@pytest.mark.parametrize("n,items,types,hidden,mnR,mnA,table_kb,virial,want", [
    (9_000, 71, 1, 30, 112, 40, 6, 1, 1), (16_000, 125, 1, 30, 136, 48, 6, 0, 0), (60_000, 469, 1, 30, 136, 48, 6, 1, 0),
    (16_000, 125, 4, 50, 24, 24, 43, 0, 0), (25_600, 200, 4, 50, 24, 24, 43, 1, 0),  # monolayer
    (25_600, 400, 4, 50, 24, 24, 43, 1, 0), (12_288, 96, 4, 50, 24, 24, 43, 1, 1),
    (25_600, 200, 3, 40, 128, 64, 26, 0, 1), (60_001, 469, 3, 40, 128, 64, 26, 1, 0),  # nanowire
    (20_000, 157, 1, 30, 328, 112, 6, 1, 1),  # many pairs
    (12_000, 94, 1, 700, 112, 40, 134, 1, 0), (9_500, 75, 1, 700, 112, 40, 134, 1, 1),  # a wide layer
    (25_600, 200, 1, 700, 112, 40, 134, 0, 1), (12_000, 94, 2, 300, 112, 40, 104, 0, 0)])
def test_evaluation_kernels_of_a_batch(host, n, items, types, hidden, mnR, mnA, table_kb, virial, want):
    args = (n, items, types, hidden, mnR, mnA, table_kb * 1024, virial)
    assert host.lib.host_by_groups(*args, 0) == want
    assert host.lib.host_by_groups(*args, 1) == 1  # FP64
