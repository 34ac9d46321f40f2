"""The library's host code without a GPU: what it allocates, uploads, launches
and captures, on the fake runtime of fake_cuda.py."""
import ctypes

import pytest

import fake_cuda


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fake_cuda.load(tmp_path_factory.mktemp("fake"))


STREAM = 0x1234


class Handle:
    def __init__(self, fake, n, nmax=20, lmax=10, precision="fp64", alpha=1.0, stream=STREAM, limit=0, offsets=None):
        from paper_2602_13385_gb300 import _lib
        c = _lib.scf_config()
        c.nmax, c.lmax, c.alpha, c.b, c.G, c.dt = nmax, lmax, alpha, 0.7, 1.0, 0.01
        c.precision = {"fp64": _lib.SCF_FP64, "mixed": _lib.SCF_MIXED}[precision]
        offsets = [0, n] if offsets is None else offsets
        self.lib, self.h = fake.lib, ctypes.c_void_p()
        fake.reset(limit)
        self.rc = fake.lib.scf_init(ctypes.byref(c), len(offsets) - 1, (ctypes.c_int64 * len(offsets))(*offsets), None,
                                    ctypes.c_void_p(stream), ctypes.byref(self.h))

    def binned(self):
        return self.lib.scf_launches_per_call(self.h, 2) > 4

    def call(self, name, *args):
        return getattr(self.lib, name)(self.h, *args)

    def __enter__(self):
        return self

    def __exit__(self, *a):
        if self.h:
            self.lib.scf_free(self.h)


def test_the_fake_runtime_sees_a_step(fake):
    with Handle(fake, 20000) as h:
        assert h.rc == 0 and h.binned()
        fake.reset()
        assert h.call("scf_step", 0x1000, 0x2000, 0x3000, None, 2) == 0
        log = fake.log()
        assert log.count(f"graph_launch {hex(STREAM)}") == 2
        assert sum("k_moments" in x for x in fake.launches()) == 1
    assert fake.used() == 0


def unordered_uploads(log, stream):
    """Uploads and clears that a launch on ``stream`` may overtake."""
    pending, bad = 0, []
    for x in log:
        w = x.split()
        if w[0] in ("copy", "copy_symbol", "memset") or w[0] in ("copy_async", "memset_async") and w[2] != hex(stream):
            pending += 1
        elif w[0] == "synchronize" and w[1] == "0x1":  # the legacy stream
            pending = 0
        elif w[0] == "launch" and pending:
            bad.append(x)
    return bad, pending


@pytest.mark.parametrize("precision,n,alpha", [("fp64", 20000, 1.0), ("fp64", 20000, 0.5), ("mixed", 100000, 1.0),
                                               ("fp64", 500, 1.0)])
def test_setup_is_ordered_before_the_kernels_that_read_it(fake, precision, n, alpha):
    """Also what the handle leaves behind: a call on its stream comes after all of it."""
    with Handle(fake, n, precision=precision, alpha=alpha) as h:
        assert h.rc == 0
        assert unordered_uploads(fake.log(), STREAM) == ([], 0)
        fake.reset()
        assert h.call("scf_set_option", 3, 64 if alpha == 1.0 else 128) == 0  # a new block map
        assert unordered_uploads(fake.log(), STREAM) == ([], 0)


@pytest.mark.parametrize("precision,n,alpha", [("fp64", 5000, 1.0), ("fp64", 5000, 0.5), ("mixed", 2000, 1.0)])
def test_sources_of_uploads_outlive_them(fake, precision, n, alpha):
    """A copy from pageable memory may read its source until the stream is waited for."""
    fake.lib.fake_forget_uploads()
    with Handle(fake, n, precision=precision, alpha=alpha) as h:
        assert h.rc == 0 and fake.lib.fake_uploads() > 10 and fake.lib.fake_lost_uploads() == 0
        assert h.call("scf_set_option", 3, 64 if alpha == 1.0 else 128) == 0
        assert h.call("scf_set_option", 2, 128) == 0
        assert fake.lib.fake_lost_uploads() == 0
        assert h.call("scf_autotune", 0x1000, None, 0x2000, 1, None) == 0
        assert fake.lib.fake_lost_uploads() == 0
        h.call("scf_retune_alpha", 0x1000, None, ctypes.c_double(0.5), ctypes.c_double(1.5), None)
        assert fake.lib.fake_lost_uploads() == 0
    fake.lib.fake_forget_uploads()


def test_setup_stays_out_of_a_capture(fake):
    with Handle(fake, 20000, stream=STREAM):  # the constants are up
        pass
    fake.capturing()
    try:
        with Handle(fake, 20000, stream=STREAM) as h:
            assert h.rc == 0 and h.binned()
            log = fake.log()
            assert not [x for x in log if hex(STREAM) in x]
            assert log[-1] == "synchronize 0x1"
    finally:
        fake.capturing(False)


def grid_of(fake, kernel):
    return [tuple(int(v) for v in x.split()[2:6]) for x in fake.log() if x.startswith("launch") and kernel in x]


@pytest.mark.parametrize("sizes,blocks,threads", [([64] * 2048, 1, 256), ([1024], 1, 256), ([1025], 1, 1024),
                                                  ([3000] * 304, 1, 1024), ([10000] * 64, 1, 1024), ([30000] * 16, 8, 1024),
                                                  ([13000], 1, 1024), ([14000, 0, 5], 8, 1024), ([200000] * 300, 1, 1024)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_blocks_of_the_selection(fake, precision, sizes, blocks, threads):
    """A cluster of blocks a progenitor only where it pays (rule in scf_escape.cu)."""
    off = [0]
    for s in sizes:
        off.append(off[-1] + s)
    with Handle(fake, 0, nmax=4, lmax=2, precision=precision, offsets=off) as h:
        assert h.rc == 0
        fake.reset()
        assert h.call("scf_bound", 0x1000, 0x2000, ctypes.c_double(0.5), ctypes.c_double(0.9), None, 0x3000, None, 0x4000) == 0
        assert grid_of(fake, "k_select") == [(blocks * len(sizes), 1, 1, threads)]


@pytest.mark.parametrize("precision,sizes,ordered", [
    ("mixed", [300], True), ("mixed", [8000], True), ("mixed", [16384], False), ("mixed", [64] * 2048, True),
    ("mixed", [700] * 2048, True), ("mixed", [1000] * 2048, False), ("mixed", [100000], False),
    ("fp64", [1000], True), ("fp64", [4096], True), ("fp64", [6000], False), ("fp64", [300] * 2048, True),
    ("fp64", [700] * 2048, False), ("fp64", [1000] * 16, True)])
def test_small_samples_take_ordered_pairs(fake, precision, sizes, ordered):
    off = [0]
    for s in sizes:
        off.append(off[-1] + s)
    with Handle(fake, 0, nmax=4, lmax=2, precision=precision, offsets=off) as h:
        fake.reset()
        assert h.call("scf_bound", 0x1000, 0x2000, ctypes.c_double(0.5), ctypes.c_double(0.9), None, 0x3000, None, 0x4000) == 0
        assert bool(grid_of(fake, "k_bound_ordered")) == ordered
        assert bool(grid_of(fake, "k_bound_pairs")) != ordered


@pytest.mark.parametrize("precision,sizes,megabytes", [("mixed", [10 ** 6], 120), ("fp64", [10 ** 6], 60),
                                                       ("mixed", [100000] * 10, 120), ("fp64", [1000] * 1024, 50)])
def test_workspace_of_the_pair_sums(fake, precision, sizes, megabytes):
    """The handle's memory without bins (lmax 2): keys, block maps, and the pair sums' slots."""
    off = [0]
    for s in sizes:
        off.append(off[-1] + s)
    with Handle(fake, 0, nmax=4, lmax=2, precision=precision, offsets=off) as h:
        assert h.rc == 0
        assert fake.used() < (megabytes + 20) * 1e6


def test_pair_sums_without_the_memory_for_their_slots(fake):
    n = 10 ** 6
    with Handle(fake, n, nmax=4, lmax=2) as h:
        full = fake.used()
    with Handle(fake, n, nmax=4, lmax=2, limit=full - 8 * n) as h:
        assert h.rc == 0 and fake.used() <= full - 8 * n
        fake.reset()
        assert h.call("scf_bound", 0x1000, 0x2000, ctypes.c_double(0.5), ctypes.c_double(0.9), None, 0x3000, None, 0x4000) == 0
        assert [g[2] for g in grid_of(fake, "k_bound_ordered")] == [1]  # one slot
        assert not [x for x in fake.log() if x.startswith("memset")]
    with Handle(fake, n, nmax=4, lmax=2, limit=full - 48 * n) as h:
        assert h.rc == -6  # out of memory


@pytest.mark.parametrize("first", ["scf_step", "scf_step_host"])
def test_a_captured_step_is_replayed_on_its_own_route_only(fake, first):
    """A mixed host step runs the direct kernels, a step over the same page-locked arrays
    the bins (here the field alone: one thread per output is chosen for kernel 1)."""
    arrays = (0x1000, 0x2000, 0x3000)
    with Handle(fake, 100000, precision="mixed") as h:
        assert h.call("scf_set_option", 2, 128) == 0
        fake.host_mapped()
        calls = {"scf_step": lambda: h.call("scf_step", *arrays, None, 1),
                 "scf_step_host": lambda: h.call("scf_step_host", None, None, None, None, *arrays, None, 8)}
        for name in sorted(calls, key=lambda c: c != first) * 2:
            fake.reset()
            fake.host_mapped()
            assert calls[name]() == 0
            bins = [k for k in fake.launches() if "k_bin" in k or "k_field" in k]
            assert fake.log().count("capture") == 1
            assert bool(bins) == (name == "scf_step"), (name, fake.launches())
        fake.reset()
        fake.host_mapped()
        assert calls[name]() == 0 and fake.log().count("capture") == 0  # the same route again: no new capture


def test_host_step_without_the_memory_for_its_device_copy(fake):
    n, arrays = 60000, (0x1000, 0x2000, 0x3000)
    with Handle(fake, n) as h:
        assert h.binned()
        for limit, binned in ((fake.used() + 1000, False), (0, True)):
            fake.reset(limit)
            fake.host_mapped()
            assert h.call("scf_step_host", None, None, None, None, *arrays, None, 8) == 0
            assert bool([k for k in fake.launches() if "k_bin" in k]) == binned
            assert h.binned()


@pytest.mark.parametrize("precision,n", [("fp64", 100000), ("mixed", 200000)])
def test_bins_give_way_to_the_workspace_that_a_handle_needs(fake, precision, n):
    with Handle(fake, n, precision=precision) as h:
        mallocs = [int(x.split()[1]) for x in fake.log() if x.startswith("malloc")]
        assert h.binned() and len(mallocs) == 2
    least = mallocs[1] - 8 * n * (mallocs[1] // (8 * n))  # at least this much without the pair sums
    ran = []
    for limit in range(sum(mallocs), least, -max(1, sum(mallocs) // 60)):
        with Handle(fake, n, precision=precision, limit=limit) as h:
            ran.append((h.rc, h.rc == 0 and h.binned()))
            if h.rc == 0:
                fake.reset()
                assert h.call("scf_step", 0x1000, 0x2000, 0x3000, None, 1) == 0
                assert bool([k for k in fake.launches() if "k_bin" in k]) == h.binned()
        assert fake.used() == 0
    kinds = [r for i, r in enumerate(ran) if i == 0 or r != ran[i - 1]]
    # with bins, then without, and only a handle that has no room for one slot is refused
    assert kinds in ([(0, True), (0, False), (-6, False)], [(0, True), (0, False)]), kinds
    assert ran.count((0, False)) * (sum(mallocs) // 60) > mallocs[0] * 0.8


def test_shared_memory_limits_are_set_once_to_the_same_value(fake):
    """A kernel's limit is not the handle's: set at the first need to what any handle may
    take, so no handle lowers it between another's set and launch, nor under its graph."""
    with Handle(fake, 60000, nmax=20, lmax=10) as a:
        first = [x for x in fake.log() if x.startswith("attribute") and "k_bin_count" in x]
        with Handle(fake, 60000, nmax=40, lmax=12, alpha=4.0) as b:  # many more bins
            limits = first + [x for x in fake.log() if x.startswith("attribute") and "k_bin_count" in x]
            assert len(set(limits)) == 1 and len(limits) == 2
            for h in (a, b):
                fake.reset()
                assert h.binned() and h.call("scf_step", 0x1000, 0x2000, 0x3000, None, 1) == 0
                assert h.call("scf_adjoint_level", 0x1000, None, ctypes.c_double(0.01), 1, 0x2000, 0x3000, None, None) in (0, -4)
                assert not [x for x in fake.log() if x.startswith("attribute") and ("k_bin" in x or "k_moments" in x)]
                smem = [int(x.split()[6]) for x in fake.log() if x.startswith("launch") and "k_bin_count" in x]
                assert smem and max(smem) <= int(limits[0].split()[-1])


@pytest.mark.parametrize("precision,n,ms,tile", [
    ("mixed", 300000, [0.2, 0.5, 0.5, 0.4, 0.1], 0),     # one thread per output beats the direct kernels, the bins beat it
    ("mixed", 300000, [0.2, 0.5, 0.5, 0.4, 0.3], 64),
    ("mixed", 300000, [0.5, 0.5, 0.5, 0.4], 0),
    ("mixed", 3000, [0.5, 0.2, 0.5, 0.4], 128),          # no bins
    ("fp64", 30000, [0.5, 0.5, 0.2], 256)])              # any tile leaves them on
def test_autotuning_does_not_drop_the_bins(fake, precision, n, ms, tile):
    with Handle(fake, n, precision=precision) as h:
        was = h.binned()
        fake.reset()
        fake.elapsed(ms)
        assert h.call("scf_autotune", 0x1000, None, 0x2000, 1, None) == 0
        got = ctypes.c_int()
        assert h.call("scf_get_option", 2, ctypes.byref(got)) == 0 and got.value == tile
        fake.reset()
        assert h.call("scf_step", 0x1000, 0x2000, 0x3000, None, 1) == 0
        assert bool([k for k in fake.launches() if "k_moments" in k]) == (was and tile != 64)


@pytest.mark.parametrize("precision,n", [("mixed", 300000), ("fp64", 20000), ("mixed", 2000)])
def test_a_step_on_new_arrays_updates_the_graph(fake, precision, n):
    with Handle(fake, n, precision=precision) as h:
        fake.reset()
        for k in (1, 2, 3):
            assert h.call("scf_step", 0x1000 * k, 0x10000 * k, 0x100000 * k, None, 1) == 0
        log = fake.log()
        assert [log.count(x) for x in ("capture", "instantiate", "update", f"graph_launch {hex(STREAM)}")] == [3, 1, 2, 3]
        assert h.call("scf_set_option", 3, 64) == 0  # another shape: another graph
        fake.reset()
        assert h.call("scf_step", 0x1000, 0x2000, 0x3000, None, 1) == 0
        assert fake.log().count("instantiate") == 1 and fake.log().count("update") == 0


@pytest.mark.parametrize("nmax,lmax,sizes,calls", [   # calls over the bins: coefficients, field, step, adjoint level
    (20, 8, [4738], "s a"), (20, 8, [23000], "cfsa"), (20, 10, [1000000], "cfsa"), (10, 5, [26000], "fsa"),
    (10, 5, [7600] * 10, "fa"), (10, 5, [14900] * 10, "fsa"), (6, 3, [84000], "a"), (6, 3, [10500] * 10, ""),
    (9, 12, [6700] * 10, "f"), (9, 12, [33000] * 10, "fsa"), (9, 12, [6900] * 64, "f"), (8, 7, [16700] * 30, "fa"),
    (20, 10, [66000, 0, 5], "cfsa")])
def test_double_precision_calls_over_the_bins(fake, nmax, lmax, sizes, calls):
    """Each call where it is the faster one over the bins (rules in scf_api.cu)."""
    off = [0]
    for s in sizes:
        off.append(off[-1] + s)
    with Handle(fake, 0, nmax=nmax, lmax=lmax, offsets=off) as h:
        assert h.rc == 0
        got = ""
        for name, args in (("scf_coeffs", (0x1000, None, 0x2000)), ("scf_forces", (0x1000, 0x2000, None, 0x3000)),
                           ("scf_step", (0x1000, 0x2000, 0x3000, None, 1)),
                           ("scf_adjoint_level", (0x1000, None, ctypes.c_double(0.01), 1, 0x2000, 0x3000, None, None))):
            fake.reset()
            assert h.call(name, *args) == 0
            over = {any(k in x for x in fake.launches()) for k in ("k_bin_count", "k_bin_scatter")}
            assert len(over) == 1
            got += name[4] if over.pop() else ""
        assert got == calls.replace(" ", "")
        assert h.call("scf_set_option", 7, 2) == 0  # every pass of a handle that has bins
        fake.reset()
        assert h.call("scf_step", 0x1000, 0x2000, 0x3000, None, 1) == 0
        assert any("k_moments" in x for x in fake.launches())
