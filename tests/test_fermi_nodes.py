"""The node tables of csrc/fermi_nodes.cuh in extended precision: every class
reproduces the grand-canonical functions to the errors that the tables are made
for, with nothing allowed for the test's own rounding (64-bit significands or
more: 1e-19 X sum a is below 1e-14)."""
import os
import re

import numpy as np
import pytest

from paper_1502_07028_gb300 import _build

LD = np.longdouble
TEXT = open(os.path.join(_build.CSRC, "fermi_nodes.cuh")).read()
CLASSES = [LD(v) for v in re.search(r"#define PTCA_FERMI_X \\\n([^\n]*)", TEXT).group(1).split(",")]


def _rows(name):
    body = TEXT.split(f"#define {name} ")[1].split("\n\n")[0].replace("\\", "")
    out = []
    for M, X, c, e, y, a, b in re.findall(r"\{(\d+), ([^,{]+), ([^,{]+), ([^,{]+),\s*\{([^}]*)\},\s*\{([^}]*)\},\s*\{([^}]*)\}\}", body):
        y, a, b = (np.array([LD(v) for v in q.split(",")]) for q in (y, a, b))
        assert y.size == a.size == b.size == int(M) and np.all(np.diff(y) < 0)
        out.append((LD(X), LD(c), LD(e), y, a, b))
    return out


@pytest.mark.skipif(np.finfo(LD).eps > 2e-19, reason="needs a long double wider than 64 bits")
@pytest.mark.parametrize("name,most,modulus,near,far", [("PTCA_FERMI_NODES", 21, 3e-7, 1.9e-6, 4e-9),
                                                        ("PTCA_FERMI_NODES_DF", 32, 6e-11, 2.5e-10, 3e-12)])
def test_every_class_holds_its_errors(name, most, modulus, near, far):
    rows = _rows(name)
    assert len(CLASSES) == 17 and [r[0] for r in rows] == CLASSES
    for X, c, e, y, a, b in rows:
        assert y.size <= most
        x = np.concatenate([np.linspace(LD(0), LD(12), 4001), np.exp(np.linspace(np.log(LD(12)), np.log(X), 8001))])
        lncosh = x / 2 + np.log1p(np.exp(-x)) - np.log(LD(2))
        fit = c + e / 2 * x ** 2
        tanh = np.zeros_like(x)
        for yj, aj, bj in zip(y, a, b):
            fit += aj / 2 * np.log1p((x / yj) ** 2)
            tanh += bj * np.arctan(x / yj)
        d = np.abs(tanh - np.tanh(x / 2) / 2)
        assert np.abs(fit - lncosh).max() <= modulus, (name, X)
        assert d.max() <= near and d[x > 14].max() <= far, (name, X, d.max())


def test_filling_errors_average_out():
    # FP32: the error is odd in x; its first two odd moments over |x| < 16 vanish
    # as well, so that a density of levels that varies slowly over 16 T sees none
    # of it (the moment of a constant error e is e)
    x = np.linspace(0.0, 16.0, 40001)
    for X, _, _, y, _, b in _rows("PTCA_FERMI_NODES"):
        err = np.arctan(x[:, None] / y.astype(float)) @ b.astype(float) - np.tanh(x / 2) / 2
        for p in (1, 3):
            w = (p + 1) * (x / 16) ** p / 16
            assert abs(np.sum((w * err)[1:] + (w * err)[:-1]) / 2 * (x[1] - x[0])) < 2e-9, (X, p)
