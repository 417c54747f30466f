"""CPU: the exact sums and float pairs of csrc/exact.cuh, built for the host with
g++ (the header's device functions also compile there), against plain integer,
FP64 and long double arithmetic over their whole windows.

The moments are exact sums and correctly rounded quotients, so no difference is
allowed.  The equilibrium pairs must keep the relative error below the 2^-42 that
eq_store guards against (2^-42.5 stated)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2503_07898_gb300", "csrc")
INCLUDE = "/usr/local/cuda/include"


@pytest.mark.skipif(not shutil.which("g++") or not os.path.isdir(INCLUDE), reason="needs g++ and the CUDA headers")
@pytest.mark.parametrize("q", [19, 27])
def test_exact_forms_on_the_host(tmp_path, q):
    exe = str(tmp_path / "exact")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", f"-DLBM_Q={q}", "-I", CSRC, "-isystem", INCLUDE,
                    os.path.join(HERE, "exact_host.cpp"), "-o", exe], check=True)
    run = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=300)
    out = {k: float(v) for k, v in (line.split() for line in run.stdout.splitlines())}
    for s in ("f32", "f16", "bf16"):
        assert out[s + "_wrong_sums"] == 0
        assert out[s + "_wrong_quotients"] == 0
        assert out[s + "_taken"] >= 300000
    assert out["wrong_round_quotient"] == 0
    assert out["equilibrium_log2_error"] < -42.5
    assert out["equilibrium_rejected"] == 0
    assert out["split_taken_outside"] == 0
    assert out["sums_taken_outside"] == 0
