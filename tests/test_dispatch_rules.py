"""Which kernel a call takes: the rules, called in the library itself.  No GPU work here."""
import ctypes
import os


def _lib():
    import __graft_entry__
    from paper_2504_13373_gb300 import gasa
    if not os.path.exists(gasa.LIB_PATH):
        __graft_entry__.build()
    return gasa.load()


def _team64_rows(n, br, bc, per_row):
    f = _lib()["_ZN4gasa11team64_rowsEiiil"]
    f.restype = ctypes.c_bool
    return f(n, br, bc, ctypes.c_int64(-2 if per_row is None else per_row * n))


def test_fp64_small_power_of_two_blocks_keep_lane_groups():
    """Blocks of fewer values than a warp has lanes take the FP64 team kernel only where no
    lane-group kernel exists for them, however long their rows."""
    for n, per_row in ((8192, 31), (2048, 75), (512, 139), (700, 30), (4000, 16)):
        assert not _team64_rows(n, 4, 4, per_row)
        assert not _team64_rows(n, 2, 8, per_row)
        assert _team64_rows(n, 5, 5, per_row)
    assert not _team64_rows(8192, 4, 10, 40) and not _team64_rows(6000, 8, 12, 20)
    assert _team64_rows(20000, 8, 8, 70) and _team64_rows(2048, 8, 8, 13)
    assert _team64_rows(4096, 12, 12, 17) and _team64_rows(300, 16, 16, None)
    assert not _team64_rows(300, 4, 4, None)
