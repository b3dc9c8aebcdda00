"""The split RK4 step's host build (tests/split_step_host.cpp): circular orbits over steps of
1e-5 to 2e-3, distances from 0.08 of the Earth and 0.002 of the Moon, several mass parameters,
are no less exact than plain FP64 steps; states come back from their words unchanged; and the
split residuals err by what the header states."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
EM, SE = 0.01215058560962404, 3.0e-6

# moon, mu, r, h, arc
CASES = [(0, EM, r, h, min(0.46, 3000 * h)) for h in (1e-5, 5e-5, 1e-4, 2.5e-4, 5e-4, 1e-3, 2e-3)
         for r in (0.08, 0.12, 0.17, 0.26, 0.36, 0.5, 0.62, 0.72, 0.8, 1.0)]
CASES += [(1, EM, r, h, 0.46 if h > 2e-4 else 0.1) for h in (1e-4, 2.5e-4, 5e-4, 1e-3, 2e-3)
          for r in (0.012, 0.02, 0.026, 0.035, 0.042, 0.05, 0.065, 0.1, 0.2)]
CASES += [(0, mu, r, 5e-4, 1.0) for mu in (SE, 0.1, 0.3) for r in (0.4, 0.6, 0.8, 0.97)]
CASES += [(1, SE, r, h, 0.46) for h in (5e-4, 1e-3) for r in (0.002, 0.003, 0.006, 0.02)]
CASES += [(1, mu, r, h, 0.46) for mu in (0.1, 0.3, 0.499) for h in (5e-4, 2e-3) for r in (0.1, 0.2, 0.4)]


@pytest.fixture(scope="module")
def result(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    exe = str(tmp_path_factory.mktemp("split") / "split")
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-w", "-I",
                    os.path.join(HERE, "..", "paper_2207_13175_gb300", "csrc"),
                    os.path.join(HERE, "split_step_host.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe] + [repr(v) for c in CASES for v in c], check=True, capture_output=True, text=True)
    return out.stdout.split()


def test_no_less_exact_than_fp64(result):
    # the FP64 implementation's own error varies by about a quarter between two such ones
    bad = [(c, float(q)) for c, q in zip(CASES, result) if not float(q) <= 1.25]
    assert not bad, bad


def test_states_come_back_from_words(result):
    assert result[len(CASES)] == "0"


def test_residual_errors(result):
    rms, most, rms_all, most_all = map(float, result[len(CASES) + 1:])
    # each residual passes about ten operations on second words, 2^-49 of angles up to pi/2
    # (below 0.1 rad) or pi: 10^0.5 2^-49 pi/2 / sqrt(3) root mean square, ten of them at most
    assert rms <= 5.1e-15 and rms_all <= 1.1e-14, (rms, rms_all)
    assert most <= 2.8e-14 and most_all <= 5.6e-14, (most, most_all)
