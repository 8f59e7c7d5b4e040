"""Which kernel a call takes: the rules, called in the library itself.  No GPU work here."""
import ctypes
import os


def _lib():
    import __graft_entry__
    from paper_2504_13373_gb300 import gasa
    if not os.path.exists(gasa.LIB_PATH):
        __graft_entry__.build()
    return gasa.load()


def _team64_split(n, br, bc, per_row):
    """(warps over a block's values, over a row's blocks, CTAs over a row) and values per lane"""
    out = [ctypes.c_int() for _ in range(4)]
    _lib()["_ZN4gasa12team64_splitEiiilPiS0_S0_S0_"](
        n, br, bc, ctypes.c_int64(-2 if per_row is None else int(per_row * n)),
        *[ctypes.byref(v) for v in out])
    es, epl, bs, cs = (v.value for v in out)
    return (es, bs, cs), epl


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
        assert n <= 1216 or _team64_rows(n, 5, 5, per_row)
    assert not _team64_rows(8192, 4, 10, 40) and not _team64_rows(6000, 8, 12, 20)
    assert _team64_rows(20000, 8, 8, 70) and _team64_rows(2048, 8, 8, 13)
    assert _team64_rows(4096, 12, 12, 17) and _team64_rows(300, 16, 16, None)
    assert not _team64_rows(300, 4, 4, None)


def test_fp64_team_split_of_small_levels():
    """A level whose rows leave an SM with less than 16 warps shares a row's blocks out down to
    one or two a warp; every split covers a block's values and fits a CTA."""
    for n, b, per_row, bs in ((256, 12, 17, 8), (64, 12, 14, 8), (576, 12, 17, 4), (1024, 12, 17, 2),
                              (4096, 12, 17, 1), (384, 10, 4, 4), (256, 9, 6, 4), (1024, 9, 7, 2),
                              (384, 17, 98, 4), (3072, 10, 5, 1), (1500, 13, 24, 2)):
        assert _team64_split(n, b, b, per_row)[0][1] == bs, (n, b, per_row)
    for br in range(1, 65, 3):
        for bc in range(1, 65, 3):
            for n in (1, 7, 150, 1216, 4096, 60000):
                for per_row in (0, 1, 5, 17, 64, 300, None):
                    (es, bs, cs), epl = _team64_split(n, br, bc, per_row)
                    assert es * epl * 32 >= br * bc and 1 <= epl <= 8
                    assert es * bs <= 16 and cs in (1, 2, 4, 8)
                    assert per_row is not None or (cs == 1 and bs <= 4)


def test_fp64_filled_ctas_keep_few_narrow_rows():
    """Few rows of narrow blocks that fill the CTA kernel's lanes take it; half-empty, wide,
    many or unknown ones take the teams."""
    for n, br, bc, per_row in ((256, 12, 12, 17), (1024, 12, 12, 17), (64, 12, 9, 40), (600, 12, 12, 80)):
        assert not _team64_rows(n, br, bc, per_row)
    for n, br, bc, per_row in ((2304, 12, 12, 17), (128, 13, 13, 53), (1296, 10, 10, 4),
                               (256, 16, 16, 27), (256, 12, 12, None)):
        assert _team64_rows(n, br, bc, per_row)


def test_fp32_low_and_short_rows_keep_a_lane_per_row():
    """FP32 blocks wider than 8: lanes on rows of blocks for low blocks and for short or few
    rows of blocks up to 15 x 15, teams on block rows elsewhere."""
    f = _lib()["_ZN4gasa12wide_by_rowsEiiiili"]
    f.restype = ctypes.c_bool

    def by_rows(op, n, br, bc, per_row):
        vw = 4 if bc % 4 == 0 else 2 if bc % 2 == 0 else 1
        return f(op, n, br, bc, ctypes.c_int64(-2 if per_row is None else per_row * n), vw)

    for op in (0, 1, 2, 4):
        for n in (64, 500, 32768):
            assert by_rows(op, n, 4, 10, 16) and by_rows(op, n, 8, 12, 10)
            assert by_rows(op, n, 1, 16, 9) and not by_rows(op, n, 4, 31, 16)
    assert by_rows(0, 500, 4, 10, None) and not by_rows(0, 500, 10, 10, None)
    for n, b, per_row in ((1000, 9, 40), (8000, 9, 12), (2000, 12, 12), (1000, 14, 28), (9000, 10, 9)):
        assert by_rows(3, n, b, b, per_row), (n, b, per_row)
    for n, b, per_row in ((256, 12, 20), (4000, 12, 20), (2000, 13, 40), (3072, 13, 25), (4000, 16, 16)):
        assert not by_rows(3, n, b, b, per_row), (n, b, per_row)
    # products of every width up to 40 have a kernel here, odd ones beyond a team's lanes too
    for bc in range(33, 41):
        for op in (0, 1, 2, 4):
            assert by_rows(op, 1000, bc, bc, 12) == (bc % 2 == 1)
    assert by_rows(4, 1024, 10, 8, 45) and by_rows(4, 2500, 22, 17, 36)
    assert not by_rows(4, 4096, 12, 12, 36) and not by_rows(4, 64, 22, 17, 90)


def test_every_smoothing_kernel_compiled_is_reached():
    """Thread-per-row smoothing kernels: the variant with two blocks in flight exists for the
    FP32 step at width 10, and the plain one everywhere else and not there."""
    import re
    import subprocess
    gasa = _lib()
    out = subprocess.run(["nm", "-C", gasa._name], capture_output=True, text=True, check=True).stdout
    found = {tuple(m.split(", ")) for m in re.findall(r"\bjacobi_kernel<([^>]*)>\(", out)}
    want = {(t, str(bs), str(mode), "true" if (t, bs, mode) == ("float", 10, 0) else "false")
            for t in ("float", "double") for bs in range(1, 17) for mode in range(4)}
    assert found == want
