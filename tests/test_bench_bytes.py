"""The bytes behind the bench's roofline figures of the arm and PSF-row passes:
the columns and rows an unaberrated bank stores, counted from the oracle's
pupils, and the sums against the DRAM traffic captured from the kernels."""
import numpy as np
import pytest

import bench
import phantom as ph


def masks(o, Y, X):
    """The binary source and detection pupils on the frequency grid."""
    ny, nx = np.fft.fftfreq(Y, o["pixel_um"])[:, None], np.fft.fftfreq(X, o["pixel_um"])[None]
    S = np.hypot(ny - o["tilt_y"] / o["lambda_um"], nx - o["tilt_x"] / o["lambda_um"]) <= o["na_ill"] / o["lambda_um"]
    P = np.hypot(ny, nx) <= o["na_det"] / o["lambda_um"]
    return S, P


@pytest.mark.parametrize("kinds", [("phase",), ("fluor",), ("phase", "absorption", "fluor")])
@pytest.mark.parametrize("kw", [dict(na_ill=0.8, tilt_x=0.05, tilt_y=-0.02), dict(na_ill=0.9), dict(na_ill=0.3, tilt_x=-0.6),
                                dict(na_ill=0.0, tilt_y=0.2)])
def test_stored_columns_hold_the_arms(kinds, kw):
    """No fewer cells than the arms need, and no more than one column of margin
    on each side of the source's."""
    Z, Y, X = 2, 64, 96
    o = ph.optics(**kw)
    S, P = masks(o, Y, X)
    axial = o["tilt_x"] == 0 and o["tilt_y"] == 0
    rows = Y // 2 + 1 if axial else Y
    need = room = 0
    if "phase" in kinds:
        kx = np.abs(np.fft.fftfreq(X, 1 / X)).astype(int)
        src = (S & P).any(0)
        det = P.any(0)
        a, b = len(set(kx[src]) if axial else np.flatnonzero(src)), len(set(kx[det]))
        need += rows * (a + b)
        room += rows * 4
    if "fluor" in kinds:
        need += (Y // 2 + 1) * len(set(np.abs(np.fft.fftfreq(X, 1 / X)).astype(int)[P.any(0)]))
    got = bench.even_arm_bytes(o, kinds, Z, Y, X)
    assert Z * need * 8 <= got <= Z * (need + room) * 8
    assert bench.bank_bytes(o, kinds, Z, Y, X)["tf_psf_rows"] == got + len(kinds) * Z * Y * (X // 2 + 1) * 8


def test_other_lengths_count_the_general_passes():
    o = ph.optics(na_ill=0.8, tilt_x=0.05)
    assert bench.bank_bytes(o, ("phase",), 4, 24, 96)["tf_arms"] == 2 * 4 * 24 * bench.band_columns(o, 96) * 8


def test_field_bytes_against_the_captured_traffic():
    """Compulsory bytes are what a kernel moves, but for re-reads and what the last
    writes leave in L2: the capture (64 tiles of other optics) has the arms at
    0.97 of them, the PSF rows at 1.04, the plane passes at 0.91 and 1.08."""
    n = bench.TILE_GRID[0] * bench.TILE_GRID[1]
    E = bench.TILE_CORE + 2 * bench.TILE_HALO
    algo = bench.field_algorithmic_bytes(ph.tile_optics(np.random.default_rng(3), n), bench.FIELD_Z, E, 1)
    for (workload, family), rec in bench.NCU_TRAFFIC.items():
        if workload == "field":
            assert 0.8 <= rec["bytes"] / algo[family] <= 1.25, (family, rec["bytes"] / algo[family])


def test_tuning_bytes_count_b_and_its_derivative_once():
    o = ph.optics(na_ill=0.8)
    Z, Y, X = bench.TUNE_SHAPE
    band = bench.band_columns(o, X)
    b = bench.tune_algorithmic_bytes(o, 2, 4)
    assert b["tf_arms"] == 2 * Z * Y * 8 * (5 * band + (band + 1))
    assert b["tf_psf_rows"] == b["tf_arms"] + 2 * 5 * Z * Y * (X // 2 + 1) * 8
