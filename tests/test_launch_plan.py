"""The model by which a call of s-steps chooses its launch shape (host arithmetic, compiled alone)."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2509_16793_gb300", "csrc")


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    """Compile and run a small host program against the model's header; returns its output lines."""
    def run(body):
        d = tmp_path_factory.mktemp("plan")
        src = d / "t.cpp"
        src.write_text('#include <cstdio>\n#include <vector>\n#include "gempic_plan.h"\n'
                       'using namespace gempic;\nint main() {\n' + body + '\nreturn 0;\n}\n')
        exe = str(d / "t")
        subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", exe], check=True)
        return subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()
    return run


def _marches(n, P, nz, lag):
    """The wavefront march by march: start after the one before it by `lag`, after the one that
    leaves its place has ended."""
    end, start = [0.0] * P, -lag
    for i in range(n):
        start = max(start + lag, end[i % P])
        end[i % P] = start + nz
    return max(end)


def test_wavefront_counts_a_partial_last_wave(host):
    cases = [(n, P, nz, lag) for n in list(range(1, 40)) + [70, 71, 78, 83, 84, 85, 200]
             for P in (1, 2, 7, 14, 16) for nz in (2, 24, 300, 1024) for lag in (4.0, 36.0)]
    body = "".join(f'printf("%.17g\\n", wavefront_slices({n}, {P}, {nz}, {lag}));\n'
                   for n, P, nz, lag in cases)
    for case, line in zip(cases, host(body)):
        assert float(line) == pytest.approx(_marches(*case), rel=1e-12), case
