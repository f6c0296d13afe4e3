"""The bench's figures for a round describe what the kernels do: k_tiles pulls
both hops in both phases and reduces no rows."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
sys.argv = sys.argv[:1]
import bench  # noqa: E402

MEDIUM = dict(n_u=1_000_000, n_v=500_000, n_a=10_000, n_e=20_000_000, n_ea=20_000_000, batch_tile=32)


class FakeAhpp:
    """100 G rows/s from tables of more than 100 MB, 150 from smaller ones."""

    @staticmethod
    def row_access_peak(table_bytes, op, device):
        assert op == "gather"
        return 100e9 if table_bytes > 100e6 else 150e9


def test_pulled_rows_against_the_measured_rates():
    r = bench.row_roofline(FakeAhpp, MEDIUM, 10, 0.01, 0, bench.pulled_rows(MEDIUM))
    assert r["rows_per_launch"] == 10 * 80_000_000
    # residues: 128 MB; t_V: 64 MB; t_A: 1.28 MB
    assert [p["table_bytes"] for p in r["parts"]] == [128_000_000, 128_000_000, 64_000_000, 1_280_000]
    assert r["frac"] == pytest.approx(10 * (40e6 / 100e9 + 40e6 / 150e9) / 0.01)


def test_tile_round_bytes_by_hand():
    nU, nV, nA = 1_000_000, 500_000, 10_000
    assert bench.tile_round_bytes(MEDIUM, 32) == 16 * 40_000_000 + 4 * (nU + nV) + 128 * (7 * nU + 2 * nV + 3 * nA)


def test_single_round_bytes_by_hand():
    nU, nV, nA = 1_000_000, 500_000, 10_000
    state = 4 * (7 * nU + 2 * nV + 3 * nA)
    rows = 4 * (nU + nV) + 4 * nU
    assert bench.q1_round_bytes(MEDIUM) == 16 * 20_000_000 + 8 * 20_000_000 + rows + state
    assert bench.q1_round_bytes(MEDIUM, bf16=False) == 16 * 20_000_000 + 16 * 20_000_000 + rows + state
    many = dict(MEDIUM, n_a=70_000)
    assert bench.q1_round_bytes(many) - bench.q1_round_bytes(MEDIUM) == 4 * 20_000_000 + 12 * 60_000
