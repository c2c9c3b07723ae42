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


# measured: ms of n s-steps of 200 slices on clusters of C CTAs, {(nx, ny, ppc, eb): {C: (shared bytes,
# marches in flight, {n: ms})}}, C ascending; the largest is the simulation's own
MEASURED_3D = {
    (64, 64, 2, 4): {4: (231680, 16, {1: 6.28, 4: 6.70, 8: 7.25, 12: 7.67, 48: 20.45}),
                     8: (141568, 15, {1: 3.42, 4: 3.62, 8: 3.92, 12: 4.10, 48: 12.99}),
                     16: (81152, 7, {1: 2.73, 4: 2.83, 8: 5.24, 12: 5.43, 48: 17.34})},
    (64, 64, 8, 4): {4: (229632, 16, {1: 11.95, 4: 12.77, 8: 13.72, 12: 14.59, 48: 39.12}),
                     8: (231680, 15, {1: 8.31, 4: 8.72, 8: 9.41, 12: 10.06, 48: 32.36}),
                     16: (179456, 7, {1: 4.54, 4: 4.60, 8: 8.83, 12: 8.88, 48: 28.61})},
    (128, 64, 1, 4): {8: (206720, 15, {1: 4.99, 4: 5.24, 8: 5.67, 12: 5.97, 48: 19.22}),
                      16: (118656, 7, {1: 3.19, 4: 3.31, 8: 6.16, 12: 6.39, 48: 20.61})},
    (128, 64, 8, 4): {8: (231296, 15, {1: 12.13, 4: 12.77, 8: 13.70, 12: 14.59, 48: 47.24}),
                      16: (232320, 7, {1: 8.69, 4: 9.10, 8: 17.00, 12: 17.63, 48: 58.91})},
    (256, 32, 2, 4): {8: (225920, 15, {1: 7.51, 4: 7.99, 8: 8.59, 12: 8.96, 48: 29.11}),
                      16: (170000, 7, {1: 5.02, 4: 5.26, 8: 9.52, 12: 9.86, 48: 32.09})},
    (32, 64, 2, 8): {4: (223000, 16, {1: 42.6, 4: 45.6, 8: 50.3, 12: 53.1, 48: 139.4}),
                     8: (137000, 15, {1: 24.2, 4: 25.8, 8: 27.9, 12: 29.3, 48: 90.1}),
                     16: (79000, 7, {1: 15.3, 4: 15.8, 8: 29.5, 12: 30.3, 48: 90.3})},
}


@pytest.mark.parametrize("grid", list(MEASURED_3D))
def test_3d_cluster_sizes_follow_the_number_of_s_steps(host, grid):
    """One launch of n s-steps takes a cluster size within 6 % of the fastest one (sizes that
    close may change places within the model's error)."""
    nx, ny, ppc, eb = grid
    sizes = MEASURED_3D[grid]
    ns = list(next(iter(sizes.values()))[2])
    body = "std::vector<ShapeTime> t;\n"
    for C, (smem, maxcl, _) in sizes.items():
        body += f"t.push_back({{slice_cycles({{{nx}, {ny}, {ppc}, {eb}, {C}, 1, 0, {smem}}}), {maxcl}}});\n"
    for n in ns:
        body += f'printf("%d\\n", pick_shape(t, {n}, 200, 4.0, 0, false).shape);\n'
    for n, line in zip(ns, host(body)):
        taken = list(sizes.values())[int(line)][2][n]
        assert taken <= 1.06 * min(v[2][n] for v in sizes.values()), n
