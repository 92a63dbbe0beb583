"""The table-driven log1p and arc tangent of kernel generation, compiled for the
host (csrc/corner_terms.cuh is plain C++ but for CUDA's qualifiers).

Bar, derived from the evaluation: the tabulated term, the constant (ln 2 or
pi / 2), the product with it, the short series and the final sum each round
once, at most 1.5 times the result in size (the series may take a third off the
tabulated term), and the series' own argument carries three more roundings of a
term below a quarter of the result: 8 units of 2^-53, relative.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2005_10160_gb300 import capi

BAR = 8 * 2.0 ** -53

SOURCE = r"""
#define __host__
#define __device__
#define __forceinline__ inline
#include <stdio.h>
#include "corner_terms.cuh"
int main(int, char** a) {
    static grav::CornerTables t;
    for (int e = 0; e < grav::CornerTables::LOGS; ++e) grav::corner_table_entry(t, e);
    FILE* in = fopen(a[1], "rb");
    FILE* out = fopen(a[2], "wb");
    double v[2], r[2];
    while (fread(v, sizeof(double), 2, in) == 2) {
        r[0] = grav::log1p_pos(v[0], t);
        r[1] = grav::atan_ratio(v[0], v[1], t);
        fwrite(r, sizeof(double), 2, out);
    }
    return fclose(out);
}
"""


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("corner")
    (d / "m.cpp").write_text(SOURCE)
    csrc = os.path.join(capi.HERE, "csrc")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", csrc, str(d / "m.cpp"), "-o", str(d / "m")], check=True)

    def run(a, b):
        np.stack([a, b], 1).tofile(d / "in")
        subprocess.run([str(d / "m"), str(d / "in"), str(d / "out")], check=True)
        return np.fromfile(d / "out").reshape(-1, 2)

    return run


@pytest.mark.parametrize("where", ["all", "intervals", "equal"])
def test_log1p_and_atan_of_ratio(evaluate, where):
    if np.finfo(np.longdouble).nmant <= 52:
        pytest.skip("no long double wider than FP64")
    rng = np.random.default_rng(3)
    if where == "all":  # twelve decades each side, and the far ends
        a = np.concatenate([10.0 ** rng.uniform(-12, 12, 20000), 10.0 ** rng.uniform(-290, 290, 2000)])
        b = np.concatenate([10.0 ** rng.uniform(-12, 12, 20000), 10.0 ** rng.uniform(-4, 4, 2000)])
    elif where == "intervals":  # a few units in the last place about every table boundary
        k, i = np.meshgrid(np.arange(-1, 40), np.arange(129))
        w = ((1.0 + i / 128.0) * 2.0 ** k).ravel()
        step = np.arange(-2, 3)[:, None]
        a = np.concatenate([(w - 1.0 + step * np.spacing(w)).ravel(), ((i.ravel() / 128.0) * (1 + step * 2.0 ** -52)).ravel()])
        a = a[a > 0]
        b = np.ones_like(a)
    else:
        a = 10.0 ** rng.uniform(-9, 9, 1000)
        b = a * (1 + rng.integers(-3, 4, 1000) * 2.0 ** -52)
    got = evaluate(a, b)
    la, lb = a.astype(np.longdouble), b.astype(np.longdouble)
    for g, ref in ((got[:, 0], np.log1p(la)), (got[:, 1], np.arctan2(la, lb))):
        err = np.abs(g.astype(np.longdouble) - ref) / ref
        worst = int(np.argmax(err))
        assert err[worst] <= BAR, (a[worst], b[worst], float(err[worst] / 2.0 ** -53))
