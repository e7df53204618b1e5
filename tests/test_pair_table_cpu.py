"""The FP64 short range's pair-function table (``csrc/pair_table.cuh``), checked on the host against
long-double erfc and exp. A double-float argument and result carry roundings of 2^-48, which reach
the value through its condition number in s = rho^2 (1/2 for the unscreened potential, 3/2 for the
force, 5/2 for the Hessian term): weighted with the pair forces of uniformly spread neighbours the
error stays below that, and for the force and the potential below the error of the double-float
functions that the table stands in for. At the ends of every row it stays below the tolerance the
fit accepts plus eight such roundings; the close-pair series keeps the bound of the double-float
functions (1e-13)."""
import json
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("tab") / "pair_table_check")
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off",
                    "-I", os.path.join(ROOT, "paper_2103_02046_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "pair_table_check.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("kappa", [0.5, 1.0, 3.0, 6.0])
def test_pair_table_accuracy(program, kappa):
    out = subprocess.run([program, repr(kappa)], check=True, capture_output=True, text=True)
    r = json.loads(out.stdout)
    assert r["fit"] and max(r["close"]) < 1e-13
    for key, condition in (("fco", 1.5), ("pot", 0.5), ("dfr", 2.5)):
        table, double_float, edge = r[key]
        assert table <= max(condition, 1.0) * 2.0 ** -48, (key, r)
        assert key == "dfr" or table <= double_float, (key, r)
        assert edge <= 2e-14 + 8 * 2.0 ** -47, (key, r)
