"""Bytes that bench.py counts for a Chebyshev step: FP32 vectors of real columns,
the same in the roofline record (per pairs of columns) and in --large (per
columns)."""
import types

import pytest

import bench


@pytest.mark.parametrize("columns", [4, 128, 256])
def test_chebyshev_step_bytes(columns):
    s = types.SimpleNamespace(n_atoms=4096, nb=69024, n_orb=16384)
    want = 4 * (16 * s.nb + s.nb + s.n_atoms + 1) + 4 * s.n_orb * columns * 4
    assert bench.algorithmic_bytes("inner32_cheb", s, columns // 2) == want
    rec = bench.roofline_for("inner32_cheb", 1.0, 10, s, columns // 2, {"hbm_gbs": 6787.2}, True, 1.0)
    assert rec["algorithmic_bytes_per_launch"] == want
    src = open(bench.__file__).read()
    assert src.count('algorithmic_bytes("inner32_cheb", s, max(panel // 2, 1))') == 1
