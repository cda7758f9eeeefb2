"""Launch logic of the library on the host, over a stand-in CUDA runtime:
a pair search one of whose launches fails leaves nothing behind that the next
one would take for its own; calls over 8x8 tiles find their list's order, made
by the prune or by themselves."""
import ctypes

import numpy as np
import pytest

import fake_cuda

N = 400
OUT_OF_MEMORY = 2
NB_OK = 0


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fake_cuda.load(tmp_path_factory.mktemp("fake"))


class Counts:
    """Stands in for the two kernels that use the column counts: k_bin, whose parameter 7
    they are, adds to them, k_col_sort clears them again."""

    def __init__(self):
        self.at_bin = []  # sum of the first counts that each k_bin found
        self.array = None

    def __call__(self, name, args):
        if "k_bin" in name:
            col_count = ctypes.cast(args[7], ctypes.POINTER(ctypes.c_void_p))[0]
            self.array = (ctypes.c_int * 4).from_address(col_count)
            self.at_bin.append(sum(self.array))
            for k in range(4):
                self.array[k] += N // 4
        elif "k_col_sort" in name:
            ctypes.memset(self.array, 0, ctypes.sizeof(self.array))


def search(lib, pl, box):
    x = np.zeros((N, 3), np.float32)
    b = np.asarray(box, np.float32)
    return lib.nb_search(pl, x.ctypes.data, b.ctypes.data, 0.8, None, None, None)


def create(lib):
    pl = ctypes.c_void_p()
    assert lib.nb_pairlist_create(ctypes.byref(pl), N, None) == NB_OK
    return pl


@pytest.mark.parametrize("memset_fails_too", [False, True])
@pytest.mark.parametrize("kernel", ["k_bin", "k_col_scatter", "k_col_sort", "k_search"])
def test_a_failed_search_leaves_no_counts(lib, kernel, memset_fails_too):
    pl = create(lib)
    counts = Counts()
    rec = fake_cuda.Recorder(lib, counts)
    assert search(lib, pl, (3, 3, 3)) == NB_OK
    assert not rec.memsets, "a search that succeeds clears its counts without a memset"
    rec.fail = lambda name: OUT_OF_MEMORY if kernel in name else 0
    rec.fail_memset = lambda: OUT_OF_MEMORY if memset_fails_too else 0
    assert search(lib, pl, (3, 3, 3)) != NB_OK
    assert b"out of memory" in lib.nb_last_error()
    if not memset_fails_too:  # also for a captured search, which is replayed without a call
        assert sum(counts.array) == 0
    rec.fail = rec.fail_memset = lambda *a: 0
    for _ in range(2):
        n_memsets = len(rec.memsets)
        assert search(lib, pl, (3, 4, 5)) == NB_OK
    assert len(rec.memsets) == n_memsets, "one clear is enough"
    assert counts.at_bin == [0] * len(counts.at_bin)
    lib.nb_pairlist_destroy(pl)


@pytest.mark.parametrize("capture", ["none", "calls", "prune"])
@pytest.mark.parametrize("sort_lists", [True, False])
def test_cluster_tiles_turned_on_after_a_prune_find_an_order(lib, sort_lists, capture):
    """The first 8x8 call orders a list whose prune did not; every call does whose order would not outlive
    it (captured) or whose list changes unseen (after a captured prune)."""
    from paper_2405_01420_gb300 import nb
    pl = create(lib)
    orders = []

    def emulate(name, args):
        if "k_forceI" in name:  # the parameter struct's seventh pointer
            orders.append(ctypes.cast(args[0], ctypes.POINTER(ctypes.c_void_p))[6])

    rec = fake_cuda.Recorder(lib, emulate)
    no_sort = 0 if sort_lists else nb.NB_FLAG_NO_LIST_SORT
    x, q, t = np.zeros((N, 3), np.float32), np.zeros(N, np.float32), np.zeros(N, np.int32)
    lj, F = np.zeros((1, 1, 2), np.float32), np.zeros((N, 3), np.float32)

    def forces():
        rec.names.clear()
        assert lib.nb_forces(pl, x.ctypes.data, q.ctypes.data, t.ctypes.data, 1, lj.ctypes.data, 0.6, 3.0,
                             F.ctypes.data, None, None) == NB_OK
        return sum("k_len_scatter" in k for k in rec.names)

    assert lib.nb_set_flags(pl, no_sort) == NB_OK
    assert search(lib, pl, (3, 3, 3)) == NB_OK
    lib.fake_capturing(capture == "prune")
    assert lib.nb_prune(pl, x.ctypes.data, 0.7, None) == NB_OK
    assert not any("k_len" in k for k in rec.names)
    lib.fake_capturing(capture == "calls")
    assert lib.nb_set_flags(pl, nb.NB_FLAG_CLUSTER_TILES | no_sort) == NB_OK
    made = [forces() for _ in range(3)]
    lib.fake_capturing(False)
    made += [forces() for _ in range(2)]
    want = {"none": [1, 0, 0, 0, 0], "calls": [1, 1, 1, 1, 0], "prune": [1, 1, 1, 1, 1]}[capture]
    assert made == (want if sort_lists else [0] * 5)
    assert [o is not None for o in orders] == [sort_lists] * 5
    lib.nb_pairlist_destroy(pl)


@pytest.mark.parametrize("cluster_tiles", [True, False])
def test_a_prune_orders_the_list_that_8x8_kernels_read(lib, cluster_tiles):
    from paper_2405_01420_gb300 import nb
    pl = create(lib)
    rec = fake_cuda.Recorder(lib)
    assert lib.nb_set_flags(pl, nb.NB_FLAG_CLUSTER_TILES if cluster_tiles else 0) == NB_OK
    assert search(lib, pl, (3, 3, 3)) == NB_OK
    x = np.zeros((N, 3), np.float32)
    assert lib.nb_prune(pl, x.ctypes.data, 0.7, None) == NB_OK
    assert any("k_len_scatter" in k for k in rec.names) == cluster_tiles
    lib.nb_pairlist_destroy(pl)
