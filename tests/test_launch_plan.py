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
        body += f"t.push_back({{slice_cycles({{{nx}, {ny}, {ppc}, {eb}, {C}, 1, 0, {smem}}}), {maxcl}, 0, 0}});\n"
    for n in ns:
        body += f'printf("%d\\n", pick_shape(t, {n}, 200, 4.0, 0, false).shape);\n'
    for n, line in zip(ns, host(body)):
        taken = list(sizes.values())[int(line)][2][n]
        assert taken <= 1.06 * min(v[2][n] for v in sizes.values()), n


# measured, 128 x 128 x 512 FP32: particles per cell -> ms of n s-steps in one launch, 7 marches in
# flight with an SM to each CTA and 14 with two CTAs per SM
MEASURED_128 = {
    1: ({7: 10.29, 8: 19.29, 14: 19.44, 21: 28.58, 28: 37.44},
        {7: 12.57, 8: 15.00, 14: 15.40, 21: 26.13, 28: 29.28}),
    2: ({7: 12.36, 8: 23.32, 14: 23.43, 21: 34.53, 28: 45.39},
        {7: 15.72, 8: 18.79, 14: 19.42, 21: 32.42, 28: 36.86}),
    4: ({7: 16.88, 8: 32.09, 14: 32.31, 21: 47.51, 28: 62.20},
        {7: 21.62, 8: 26.15, 14: 27.13, 21: 45.00, 28: 51.53}),
    8: ({7: 25.83, 8: 49.19, 14: 49.74, 21: 73.43, 28: 96.54},
        {7: 33.33, 8: 40.77, 14: 43.86, 21: 72.20, 28: 84.21}),
    16: ({7: 43.75, 8: 83.26, 14: 84.45, 21: 124.59, 28: 164.17},
         {7: 59.47, 8: 72.85, 14: 81.54, 21: 134.30, 28: 157.04}),
}


@pytest.mark.parametrize("ppc", list(MEASURED_128))
def test_two_ctas_per_sm_where_they_are_faster(host, ppc):
    """A call, whole waves and the rest apart, takes no longer than the faster shape in one launch."""
    shapes = "std::vector<ShapeTime> t;\n"
    for dense, maxcl in ((0, 7), (1, 14)):
        shapes += (f"SliceWork w{dense}{{128, 128, {ppc}, 4, 16, 1, {dense}, 0}};\n"
                   f"t.push_back({{slice_cycles(w{dense}), {maxcl}, slice_cycles(w{dense}, false), 7}});\n")
    for n in MEASURED_128[ppc][0]:
        ms = 0.0
        for line in host(shapes + f"for (int n = {n}; n > 0;) {{\n"
                         "Pick k = pick_shape(t, n, 512, 4.0, 0, true);\n"
                         'printf("%d %d\\n", k.shape, k.count);\nn -= k.count;\n}'):
            shape, count = map(int, line.split())
            ms += MEASURED_128[ppc][shape][count]
        assert ms <= 1.02 * min(v[n] for v in MEASURED_128[ppc]), n


# measured, 128 x 128 FP32 on short windows: (particles per cell, nz) -> ms of 8, 10 and 14 s-steps
SHORT_128 = {
    (1, 100): ({8: 3.741, 10: 3.790, 14: 4.000}, {8: 3.249, 10: 3.408, 14: 3.819}),
    (2, 100): ({8: 4.527, 10: 4.625, 14: 4.860}, {8: 4.089, 10: 4.282, 14: 4.796}),
    (8, 100): ({8: 9.504, 10: 9.713, 14: 10.390}, {8: 8.964, 10: 9.467, 14: 10.795}),
    (16, 100): ({8: 16.090, 10: 16.484, 14: 17.726}, {8: 15.835, 10: 17.201, 14: 19.830}),
    (16, 150): ({8: 24.290, 10: 24.646, 14: 25.615}, {8: 22.679, 10: 24.386, 14: 27.166}),
    (16, 250): ({8: 40.356, 10: 41.061, 14: 41.838}, {8: 36.271, 10: 38.679, 14: 42.082}),
}


@pytest.mark.parametrize("ppc,nz", list(SHORT_128))
def test_two_ctas_per_sm_on_short_windows(host, ppc, nz):
    body = "std::vector<ShapeTime> t;\n"
    for dense, maxcl in ((0, 7), (1, 14)):
        body += (f"SliceWork w{dense}{{128, 128, {ppc}, 4, 16, 1, {dense}, 0}};\n"
                 f"t.push_back({{slice_cycles(w{dense}), {maxcl}, slice_cycles(w{dense}, false), 7}});\n")
    for n in (8, 10, 14):
        body += f'printf("%d\\n", pick_shape(t, {n}, {nz}, 4.0, 0, false).shape);\n'
    for n, line in zip((8, 10, 14), host(body)):
        both = [v[n] for v in SHORT_128[ppc, nz]]
        assert both[int(line)] <= 1.05 * min(both), n


def test_ring_levels_leave_room(host):
    """Deeper wavefronts take 16 GiB and a sixteenth of the free memory at most."""
    gib = float(1 << 30)
    cases = [(0.74e9, 280e9, 23), (0.74e9, 200e9, 16), (0.74e9, 100e9, 8), (0.74e9, 8e9, 0),
             (1e6, 280e9, 128), (2 * gib, 1000 * gib, 8), (2 * gib, 16 * gib, 0)]
    out = host("".join(f'printf("%d\\n", ring_levels({a}, {b}));\n' for a, b, _ in cases))
    assert [int(v) for v in out] == [c for _, _, c in cases]
