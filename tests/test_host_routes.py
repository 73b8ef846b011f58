"""Host routes without a GPU: workspaces, launches and error returns of the
library's own host code over the stand-in runtime (host_library.py)."""
import ctypes

import pytest

import host_library

I16, F32 = 0, 1


@pytest.fixture()
def H(tmp_path):
    return host_library.load(tmp_path)


# ---------------------------------------------------------------- workspaces
@pytest.mark.parametrize("n", [64, 513, 2048, 4096, 8192, 16385, 65536])
def test_every_route_of_one_size_uses_one_workspace(H, n):
    """A fit captured in a graph keeps the workspace's address: later fits of the same n by another route (with
    statistics, an order statistic below n / 8) neither move nor free the buffer, and all of them fit in it while
    streams are being captured."""
    assert H.fit_bnb(n) == 0
    frees, held = H.lib.fake_frees(), H.lib.fake_held()
    H.set("capturing", 1)
    assert H.fit_bnb(n, h=max(1, n // 16)) == 0
    assert H.fit_bnb(n, stats=True) == 0
    assert H.fit_bnb(n) == 0
    assert (H.lib.fake_frees(), H.lib.fake_held()) == (frees, held)


@pytest.mark.parametrize("n,dtype", [(513, I16), (2048, I16), (8192, I16), (16385, I16), (64, F32), (2048, F32),
                                     (4096, F32)])
def test_auto_and_sweep_use_one_workspace(H, n, dtype):
    assert H.fit(n, dtype=dtype) == 0
    frees = H.lib.fake_frees()
    H.set("capturing", 1)
    for h in (0, max(1, n // 16)):
        assert H.fit(n, h, dtype=dtype) == 0
        assert H.fit(n, h, "sweep", dtype=dtype) == 0
    assert H.lib.fake_frees() == frees


@pytest.mark.parametrize("n,dtype,algorithm", [(600, I16, "auto"), (8192, I16, "auto"), (64, I16, "bnb"),
                                               (8192, I16, "bnb"), (2048, F32, "auto")])
def test_installed_workspace(H, n, dtype, algorithm):
    """lms_workspace_size bytes are enough for every route; less than the fit's share of them is refused by all."""
    size = H.workspace_size(n, dtype, algorithm)
    staging = 2 * ((n * (4 if dtype == F32 else 2) + 255) // 256 * 256)
    buf = ctypes.create_string_buffer(size)
    runs = [lambda: H.fit(n, 0, algorithm, dtype), lambda: H.fit(n, 1, algorithm, dtype)]
    if algorithm == "bnb":
        runs += [lambda: H.fit_bnb(n), lambda: H.fit_bnb(n, stats=True)]
    H.set_workspace(buf, size)
    assert H.fit(n, 0, algorithm, dtype, host=True) == 0
    assert [r() for r in runs] == [0] * len(runs)
    H.set_workspace(buf, size - staging - 1)
    assert [r() for r in runs] == [6] * len(runs)   # LMS_ERR_WORKSPACE


# ---------------------------------------------------------------- shared-memory limits
def test_shared_memory_limits_are_only_raised(H):
    """The limit of a kernel is shared by all host threads: a smaller call between another thread's limit and its
    launch must not lower it (plans of different sizes, fits of different n)."""
    sizes = {}

    def calls():
        for n in (4096, 600):
            assert H.fit(n) == 0 and H.fit(n, 0, "sweep") == 0 and H.fit_bnb(n, stats=True) == 0
            assert H.fit(n, dtype=F32) == 0
            rc, plan, off = H.plan([n, n])
            assert rc == 0 and H.fit_batched(plan, off) == 0
            yield n
            H.lib.lms_batch_plan_destroy(plan)

    for n in calls():
        limits = {k: H.lib.fake_limit(k.encode()) for k in set(H.kernels())}
        for k, v in limits.items():
            assert v >= sizes.get(k, 0), (n, k)
        sizes.update(limits)
    assert max(sizes.values()) > 48 * 1024


# ---------------------------------------------------------------- routes
def route(names):
    """What a call's kernels are: the one kernel, the sweep's, the staged branch-and-bound's, the plain ones."""
    parts = {"one": "k_direct", "sweep": "k_sweep", "staged": "k_node_lb", "plain": "k_plain"}
    return {k for k, part in parts.items() if any(part in n for n in names)}


@pytest.mark.parametrize("knob,value", [("clusters", 0), ("refuse_clusters", 1)])
def test_no_room_for_the_cluster(H, knob, value):
    """A device that cannot hold the one kernel's cluster, or a launch it refuses: the fits take the paths of many
    kernels."""
    H.set(knob, value)
    for call, want in ((lambda: H.fit(2048), {"sweep"}), (lambda: H.fit(8192, host=True), {"sweep"}),
                       (lambda: H.fit(2048, dtype=F32), {"sweep"}), (lambda: H.fit_bnb(2048), {"staged", "sweep"}),
                       (lambda: H.fit_bnb(65536), {"staged", "sweep"})):
        assert call() == 0
        assert route(H.kernels()) == want
    H.set("clusters", 8)
    H.set("refuse_clusters", 0)


def test_sweep_options_take_the_sweep(H):
    assert H.fit(2048) == 0 and route(H.kernels()) == {"one"}
    for opt in ({"sweepers": 100}, {"buckets": 64}):
        assert H.fit(2048, **opt) == 0 and route(H.kernels()) == {"sweep"}
        assert H.fit(2048, dtype=F32, **opt) == 0 and route(H.kernels()) == {"sweep"}


# default: plain, then the one kernel up to 4096 points (its sets of up to 256 points followed by the plain kernels,
# which pass over what it has fitted), staged above; options are kept to
@pytest.mark.parametrize("options,want", [
    ({}, {64: "plain", 96: "plain", 97: "one", 256: "one", 400: "one", 512: "one", 4096: "one", 4097: "staged"}),
    ({"plain_max_n": 128}, {64: "plain", 128: "plain", 256: "one", 512: "one", 4097: "staged"}),
    ({"plain_max_n": 256}, {256: "plain", 400: "one", 4096: "one"}),
    ({"bnb_min_n": -1}, {256: "plain", 257: "sweep", 4096: "sweep", 4097: "sweep"}),
    ({"bnb_min_n": 512}, {256: "plain", 400: "sweep", 511: "sweep", 512: "one", 4097: "staged"}),
    ({"plain_max_n": 64, "bnb_min_n": 600}, {64: "plain", 100: "sweep", 599: "sweep", 600: "one", 5000: "staged"})])
def test_batch_options_choose_the_path(H, options, want):
    for n, path in want.items():
        rc, plan, off = H.plan([n], **options)
        assert rc == 0 and H.fit_batched(plan, off) == 0
        got = route(H.kernels())
        if path == "one" and n <= 256:
            got.discard("plain")
        assert got == ({"staged", "sweep"} if path == "staged" else {path}), (n, options)
        H.lib.lms_batch_plan_destroy(plan)


def test_batch_without_room_for_the_one_kernel(H):
    H.set("no_blocks", 1)
    rc, plan, off = H.plan([64, 200, 300, 2000])
    assert rc == 0 and H.fit_batched(plan, off) == 0
    assert route(H.kernels()) == {"plain", "staged", "sweep"}
    H.set("no_blocks", 0)
