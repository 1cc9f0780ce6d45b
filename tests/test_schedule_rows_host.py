"""The schedule table's row passes at 384 points (rows of 768 samples): the
engine that runs by default is the one reported, and either can be chosen.
No GPU: the table is host state."""
import pytest

from paper_2412_09775_gb300.build import build


@pytest.fixture(scope="module")
def B():
    build()
    from paper_2412_09775_gb300 import binding
    return binding


@pytest.mark.parametrize("n", [384, 512])
def test_rows_engine_is_reported_and_can_be_pinned(B, n):
    try:
        assert B.wo_schedule_get(B.WO_PASS_ROWS, n) == B.WO_ENGINE_HYBRID
        for e in (B.WO_ENGINE_SMEM, B.WO_ENGINE_HYBRID):
            B.wo_schedule_set(B.WO_PASS_ROWS, n, e)
            assert B.wo_schedule_get(B.WO_PASS_ROWS, n) == e
    finally:
        B.wo_schedule_set(B.WO_PASS_ROWS, n, B.WO_ENGINE_DEFAULT)
    assert B.wo_schedule_get(B.WO_PASS_ROWS, n) == B.WO_ENGINE_HYBRID
    with pytest.raises(B.WoError):
        B.wo_schedule_set(B.WO_PASS_ROWS, 768, B.WO_ENGINE_HYBRID)


def test_field_tiles_of_768_stay_refused(B):
    """The passes that read tiles in place have no 384-point form."""
    assert B._lib.wo_reconstruct_field_tiles(1 << 20, 1, 1 << 20, 1, 1, 1, 768, 0, None, None, 0, 0, 1 << 20, 1 << 20,
                                             1 << 40, None) == B.STATUS_CODES["WO_ERR_UNSUPPORTED_SIZE"]
