"""The printed float64 roofline counts the operations that run on the FP64 pipe."""
import importlib
import os
import sys
import types

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_headline_fraction_is_of_the_fp64_pipe():
    sys.path.insert(0, ROOT)
    bench = importlib.import_module("bench")
    info = types.SimpleNamespace(n_fields=7, n_nodes=16_384_000, launches_per_stage=2)
    hbm = bench._roofline(info, 8, 0.5, 10, 6705.5, "measured", (None, None))
    r = bench.fp64_alu_roofline(info, {"dim": 3, "order": 4, "rain": 1}, 0.28, 10, 152, 2070.0, 1.25, hbm)
    h = bench.fp64_pipe_headline(r)
    assert r["frac"] > 1.0                                   # with the integer items it is no fraction
    items = r["flops_per_node_items"]
    rest = sum(v for k, v in items.items() if k not in bench.INTEGER_PIPE_ITEMS)
    assert h["achieved"] == pytest.approx(rest * info.n_nodes / (0.28 / 40) / 1e12)
    assert h["frac"] == pytest.approx(h["achieved"] / h["peak"]) and h["frac"] < 1.0
    assert h["all_items"]["achieved"] == r["achieved"]
    assert h["fp64_fma_probe"]["frac_of_probe"] == pytest.approx(h["achieved"] / 1.25)
