"""The FP64 walk's table of the short-range factor: committed entries equal the
generator's, and the piecewise polynomial evaluated in FP64 in the kernel's
order stays within its rounding (each of the seven operations half an ulp of a
value no larger than 1) of f(u) = erfc(u) + (2 u / sqrt(pi)) exp(-u^2)."""
import importlib.util
import os
import re
import sys

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_17145_gb300", "csrc")


def _table():
    text = open(os.path.join(CSRC, "short_range_table.inc")).read()
    n = int(re.search(r"#define OG_SR_TABLE_N (\d+)", text).group(1))
    per_unit = int(re.search(r"#define OG_SR_TABLE_PER_UNIT (\d+)", text).group(1))
    body = text[text.index("= {") + 3:text.index("};")]
    v = np.array([float(x) for x in re.findall(r"-?\d[\d.]*(?:e-?\d+)?", body)])
    return v.reshape(n, 8), per_unit


def test_table_is_what_the_generator_writes():
    pytest.importorskip("mpmath")
    spec = importlib.util.spec_from_file_location("fit_short_range_table", os.path.join(CSRC, "fit_short_range_table.py"))
    mod = importlib.util.module_from_spec(spec)
    keep, sys.dont_write_bytecode = sys.dont_write_bytecode, True
    try:
        spec.loader.exec_module(mod)
    finally:
        sys.dont_write_bytecode = keep
    assert np.array_equal(np.array(mod.entries()), _table()[0])


def test_table_accuracy_on_the_cut_interval():
    mp = pytest.importorskip("mpmath")
    v, per_unit = _table()
    assert v.shape[0] == 2.25 * per_unit
    rng = np.random.default_rng(3)
    u = np.concatenate([rng.random(1500) * 2.25, np.arange(v.shape[0]) / per_unit, [np.nextafter(2.25, 0.0)]])
    e = v[(u * per_unit).astype(int)]
    x = u - e[:, 0]
    p = e[:, 7]
    for k in range(6, 0, -1):
        p = p * x + e[:, k]
    with mp.workdps(30):
        ref = np.array([float(mp.erfc(a) + 2 * mp.mpf(a) / mp.sqrt(mp.pi) * mp.exp(-mp.mpf(a) ** 2)) for a in u])
    assert np.abs(p - ref).max() <= 7 * 2.0 ** -53
