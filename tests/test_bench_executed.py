"""CPU check of bench.py's share of executed work: instructions of the row
patterns' terms over the pipe's rate, which no hardware exceeds, against the
worked figures of the 3-wavelength cube."""
import importlib.util
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parents[1]


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_executed_under_test", ROOT / "bench.py")
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def test_executed_share(bench):
    # 3.0 M terms, 1 729 products in 28.2 ms: 24 FP32 instructions a term at 152 x 128 lanes x 2.07 GHz
    rate, peak, share = bench.executed_share("df", 3_000_000, 1, 1729, 28.2e-3)
    assert peak == pytest.approx(152 * 128 * 2.07e9 / 1e12)
    assert rate == pytest.approx(3e6 * 24 * 1729 / 28.2e-3 / 1e12)
    assert share == pytest.approx(rate / peak) and share < 1
    # FP64: two FMA a term at a 64th of the rate
    rate, peak, share = bench.executed_share("fp64", 3_000_000, 1, 1608, 48.9e-3)
    assert peak == pytest.approx(152 * 2 * 2.07e9 / 1e12) and rate == pytest.approx(3e6 * 2 * 1608 / 48.9e-3 / 1e12)
    assert bench.executed_share("mixed", 3_000_000, 4, 10, 1.0)[0] == pytest.approx(3e6 * 2 * 4 * 10 / 1e12)
    assert bench.executed_share("df", 1, 1, 1, 0.0)[0] is None
