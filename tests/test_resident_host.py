"""Argument checks of the resident solves' test hook, without a GPU."""


def test_wait_limits_need_one_object():
    from paper_2408_03452_gb300 import build, tpfa
    build.build()
    L = tpfa.lib()
    assert L.tpfa_resident_wait_limits(None, None, 1, 1) == tpfa.EINVAL
