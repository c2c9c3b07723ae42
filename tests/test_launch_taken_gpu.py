"""Which launch a call of s-steps takes, and that the taken ones agree: every case states the shape
it is there for (Sim.last_launch) next to its results."""
import numpy as np
import pytest

from paper_2509_16793_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2509_16793_gb300 import build, gempic
    build.build()
    return gempic


def _lwfa(nz, ppc=2, a0=1.0, **kw):
    w = W.lwfa_3d_128x128x1024()
    return w.with_(nzeta=nz, species=[W.Species(-1.0, 1.0, w.species[0].density, ppc)],
                   laser=W.Laser(**{**w.laser.__dict__, "a0": a0, "zeta_center": 0.5 * nz * w.h}), **kw)


def _two_ctas_per_sm(sim):
    """128 x 128 marches are 16 CTAs of 512 threads, or (two CTAs per SM) of 256."""
    t = sim.last_launch()
    assert t["march_ctas"] == 16 and t["threads"] in (256, 512)
    return t["threads"] == 256


# the diagnostics are FP32 sums over each thread's particles, added in FP64: other threads, other
# groups of at most 16 slices' particles a thread, so the last bits differ
DIAG_RTOL = 1e-5


def _same_bits(a, b):
    assert np.array_equal(a.state(), b.state())
    assert np.array_equal(a.onaxis_ez(), b.onaxis_ez())
    da, db = a.diagnostics(), b.diagnostics()
    for k in ("n_trapped", "n_stored", "n_rejoined", "pushes", "step"):
        assert da[k] == db[k], k
    for k in ("field_energy", "kinetic_energy"):
        assert abs(da[k] - db[k]) <= DIAG_RTOL * abs(db[k]), k


def test_before_any_launch(G):
    with G.Sim(W.small_2d(nzeta=16)) as s:
        with pytest.raises(G.GempicError):
            s.last_launch()
        s.step(1)
        assert s.last_launch()["in_flight"] == 1


# particles beyond the free-slot stack (ppc 5: 5120 fresh slots a CTA), a strong laser, a density
# channel; the plain runs of this grid never store a particle, so the bits are equal
@pytest.mark.parametrize("nz,ppc,a0,n,channel", [(240, 5, 1.0, 14, None), (240, 1, 1.5, 14, None),
                                                 (200, 2, 1.0, 10, (0.25, 20.0)),
                                                 (220, 8, 0.5, 9, None)])
def test_dense_march_equals_single_steps(G, nz, ppc, a0, n, channel):
    w = _lwfa(nz, ppc, a0)
    if channel:
        w = w.with_(channel=W.Channel(*channel))
    with G.Sim(w) as a, G.Sim(w) as b:
        a.step(n)
        assert _two_ctas_per_sm(a) and a.last_launch()["in_flight"] == n
        for _ in range(n):
            b.step(1)
            assert not _two_ctas_per_sm(b)
        _same_bits(a, b)


@pytest.mark.parametrize("nz,n", [(260, 14), (520, 17)])
def test_dense_march_keeps_snapshot_and_current(G, nz, n):
    """Fields and currents of the last s-step: in the dense launch itself (14), and where the call
    goes on in a second launch (17)."""
    w = _lwfa(nz, 2, 1.0, snapshot=True, capture_current=True)
    with G.Sim(w) as a, G.Sim(w) as b:
        launches = a.launch_count()
        a.step(0)
        init = a.launch_count() - launches
        a.step(n)
        assert a.launch_count() - launches - init == (1 if n == 14 else 2)
        assert _two_ctas_per_sm(a) == (n == 14)
        for _ in range(n):
            b.step(1)
        _same_bits(a, b)
        for f in ("Ex", "Ez", "Bz", "jx", "jy", "jz"):
            assert np.array_equal(a.fields(f), b.fields(f)), f
        assert np.array_equal(a.current(), b.current())


def _runs_apart(sims, n):
    """(state of the first, largest difference among the others) of simulations of one workload: the
    first does n s-steps in one call, the others one at a time.  Stored particles deposit by FP32
    reductions in global memory in whatever order they come, which the plasma then amplifies: two
    runs of the same launches differ, and the spread of three says by how much."""
    sims[0].step(n)
    for s in sims[1:]:
        for _ in range(n):
            s.step(1)
        assert not _two_ctas_per_sm(s)
    st = [s.state() for s in sims[1:]]
    return st[0], max(np.abs(x - y).max() for i, x in enumerate(st) for y in st[:i])


def test_dense_march_with_a_bunch(G):
    """A bunch of more particles per slab than threads (the window of the fields), pushed, appended
    and deposited by dense marches, is no further from single steps than 4 times as far as those
    are from each other."""
    w = W.pwfa_3d_128x128x768(n_macro=1 << 15)
    w = w.with_(nzeta=240, beam=W.Beam(**{**w.beam.__dict__, "n_peak": 0.05, "zeta_center": 120 * w.h,
                                          "sigma_z": 0.4}))
    with G.Sim(w) as a, G.Sim(w) as b, G.Sim(w) as c, G.Sim(w) as d:
        ref, apart = _runs_apart((a, b, c, d), 14)
        assert _two_ctas_per_sm(a)
        assert 0 < apart <= 1e-2 * np.abs(ref).max()
        assert np.abs(a.state() - ref).max() <= 4 * apart
        da, db = a.diagnostics(), b.diagnostics()
        assert da["n_stored"] == db["n_stored"] > 20000 and da["pushes"] == db["pushes"]
        assert abs(da["field_energy"] - db["field_energy"]) <= 1e-3 * db["field_energy"]


def test_dense_march_with_rejoining_particles(G):
    """A slow bunch: its particles (v_z = 0.75, budgets used up after some 17 slices) rejoin the
    streaming ones in every s-step, in the dense march's slots.  A budget that ends within rounding
    of a slice may end in its neighbour: 1 % of the counts."""
    w = W.pwfa_3d_128x128x768(n_macro=1 << 12)
    w = w.with_(nzeta=240, delta=1.0,
                beam=W.Beam(**{**w.beam.__dict__, "n_peak": 0.01, "zeta_center": 220 * w.h,
                               "sigma_z": 0.1, "gamma": 1.5, "rel_spread": 0.1}))
    with G.Sim(w) as a, G.Sim(w) as b, G.Sim(w) as c, G.Sim(w) as d:
        ref, apart = _runs_apart((a, b, c, d), 9)
        assert _two_ctas_per_sm(a) and a.last_launch()["in_flight"] == 9
        da, db = a.diagnostics(), b.diagnostics()
        for k in ("n_trapped", "n_stored", "n_rejoined"):
            assert db[k] > 1000 and abs(da[k] - db[k]) <= 2 + db[k] // 100, k
        assert np.abs(a.state() - ref).max() <= 4 * apart + 1e-6 * np.abs(ref).max()


@pytest.mark.parametrize("nz,n", [(800, 14), (901, 10)])
def test_dense_streamed_equals_single_steps(G, nz, n):
    import torch
    w = _lwfa(nz)
    with G.Sim(w) as a, G.Sim(w) as b:
        host = torch.empty(a.state_shape(), dtype=torch.complex64, pin_memory=True).numpy()
        host[...] = a.state()
        a.step_streamed(n, host)
        assert _two_ctas_per_sm(a)
        for _ in range(n):
            b.step(1)
        assert np.array_equal(host, b.state())
        _same_bits(a, b)


def test_streamed_2d_with_many_marches(G):
    """More than 16 streamed 2-D s-steps in flight."""
    import torch
    w = W.small_2d(nx=64, nzeta=300, ppc=2, precision=32, a0=0.5, delta=5.0)
    with G.Sim(w) as a, G.Sim(w) as b:
        host = torch.empty(a.state_shape(), dtype=torch.complex64, pin_memory=True).numpy()
        host[...] = a.state()
        a.step_streamed(40, host)
        assert a.last_launch()["in_flight"] > 16 and a.last_launch()["march_ctas"] == 1
        for _ in range(40):
            b.step(1)
        assert np.array_equal(host, b.state())


@pytest.mark.parametrize("option", ["trapping", "gt1", "beam"])
def test_split_fp32_marches_with_stored_particles(G, option):
    """FP32 marches whose particles several CTAs share, with stored particles, against the FP64
    march of one CTA: as far from it as the FP32 march of one CTA is, to a factor of 10 (both are
    FP32 runs of the same scheme, with the reductions of the stored particles in another order)."""
    kw = {"trapping": dict(delta=3.0), "gt1": dict(particle_law="GT1", delta=8.0),
          "beam": dict(beam=W.Beam(n_peak=0.002, sigma_r=3.0, sigma_z=1.5, zeta_center=8.0,
                                   gamma=200.0, n_macro=500))}[option]
    states = []
    for prec, ctas in ((64, 1), (32, 1), (32, 0)):
        w = W.small_2d(nx=128, nzeta=50, ppc=4, precision=prec, a0=2.0, delta=20.0).with_(**kw)
        with G.Sim(w, cluster_ctas=ctas, bucket_capacity=4096) as s:
            s.step(1)
            assert (s.last_launch()["march_ctas"] > 1) == (ctas == 0)
            s.step(1)
            d = s.diagnostics()
            assert d["n_stored"] + d["n_trapped"] > 0
            states.append(s.state().astype(np.complex128))
    ref, one, split = states
    for part in (slice(0, 4), slice(4, 6)):
        own = np.abs(one[part] - ref[part]).max()
        assert np.abs(split[part] - ref[part]).max() <= 10.0 * own


@pytest.mark.parametrize("nx,ny,ppc,precision", [(64, 64, 2, 32), (128, 64, 1, 32), (64, 128, 3, 32),
                                                 (64, 64, 2, 64)])
def test_3d_cluster_sizes_agree(G, nx, ny, ppc, precision):
    """Calls of many s-steps march on smaller clusters than single ones, streamed ones as well; the
    state and the stored set pass from one to the other.  The sums of a halo row's fixed-point
    currents are converted to FP32 band by band: one rounding more or less for a node and slice
    (6e-8), of which a state value takes up some hundred."""
    import torch
    w = W.small_3d(nx=nx, ny=ny, nzeta=120, ppc=ppc, precision=precision, a0=1.0)
    tol = 1e-5 if precision == 32 else 1e-11
    with G.Sim(w) as a, G.Sim(w) as b:
        for _ in range(2):                           # 15 together, one alone: there and back
            a.step(15)
            many = a.last_launch()
            a.step(1)
            assert many["march_ctas"] < a.last_launch()["march_ctas"] == a.launch_shape()["cluster_ctas"]
            for _ in range(16):
                b.step(1)
            ra, rb = a.state(), b.state()
            for part in (slice(0, 4), slice(4, 6)):
                assert np.abs(ra[part] - rb[part]).max() <= tol * np.abs(rb[part]).max()
            da, db = a.diagnostics(), b.diagnostics()
            for k in ("n_trapped", "n_stored", "n_rejoined", "pushes", "step"):
                assert da[k] == db[k], k
        host = torch.empty(a.state_shape(), pin_memory=True,
                           dtype=torch.complex128 if precision == 64 else torch.complex64).numpy()
        host[...] = a.state()
        d = a.step_streamed(12, host)
        for i in range(12):
            b.step(1)
            assert d[i]["pushes"] == b.diagnostics()["pushes"]
        rb = b.state()
        for part in (slice(0, 4), slice(4, 6)):
            assert np.abs(host[part] - rb[part]).max() <= 2 * tol * np.abs(rb[part]).max()


def test_denoised_chain_leaves_the_net_half_of_the_chip(G):
    """64 x 128: rows that the net gathers.  A chain of several s-steps marches on clusters of 8,
    one s-step (two marches) on 16; both give the same, to what a last bit of the currents can do:
    a BF16 rounding of the net (2^-8) at single voxels, in a correction of a tenth of the current."""
    import torch
    from oracle import denoise_ref as D
    w = W.small_3d(nx=64, ny=128, nzeta=96, ppc=1, precision=32, a0=0.5)
    scale = abs(w.species[0].charge * w.species[0].density)
    with G.Denoiser(G.denoiser_params_to_vector(D.init_params(seed=9, scale3=0.05)), scale) as d, \
            G.Sim(w) as a, G.Sim(w) as b:
        a.set_denoiser(d)
        b.set_denoiser(d)
        a.step(5)
        assert a.last_launch() == dict(march_ctas=8, threads=512, in_flight=7)
        for _ in range(5):
            b.step(1)
            assert b.last_launch()["march_ctas"] == 16
        sa, sb = a.state(), b.state()
        assert np.abs(sa - sb).max() <= 4e-4 * np.abs(sb).max()
        da, db = a.diagnostics(), b.diagnostics()
        for k in ("n_trapped", "n_stored", "n_rejoined", "pushes", "step"):
            assert da[k] == db[k], k
        assert abs(da["field_energy"] - db["field_energy"]) <= 4e-4 * db["field_energy"]


def test_a_full_device_takes_the_former_depth(G):
    """With less memory free than sixteen times the rings of 14 s-steps in flight (11.8 GB) a
    128 x 128 x 1024 simulation takes those of 7, and is not refused."""
    import torch
    w = W.lwfa_3d_128x128x1024()
    free, _ = torch.cuda.mem_get_info()
    ballast = torch.empty(int(free - 90e9), dtype=torch.uint8, device="cuda")
    try:
        before, _ = torch.cuda.mem_get_info()
        with G.Sim(w) as s:
            assert before - torch.cuda.mem_get_info()[0] < 10e9
            s.step(14)
            assert not _two_ctas_per_sm(s) and s.last_launch()["in_flight"] == 7
    finally:
        del ballast
        torch.cuda.empty_cache()


@pytest.mark.parametrize("option", ["refined", "residual"])
def test_128_options_of_the_generic_kernel(G, option):
    """Runs whose options the two-CTA march does not have take the generic one for any number of
    s-steps, and give what single s-steps give."""
    w = _lwfa(60)
    w = w.with_(**{"refined": dict(hz=W.refined_h(w.nzeta, w.h, 2.0)),
                   "residual": dict(residual=True)}[option])
    with G.Sim(w) as a, G.Sim(w) as b:
        a.step(14)
        assert not _two_ctas_per_sm(a)
        for _ in range(14):
            b.step(1)
        _same_bits(a, b)
        if option == "residual":
            da, db = a.diagnostics(), b.diagnostics()
            assert abs(da["gauss_residual"] - db["gauss_residual"]) <= DIAG_RTOL * db["gauss_residual"]


def test_128_gt1_takes_the_generic_kernel(G):
    """(A GT1 run's stops amplify rounding: no comparison of many s-steps.)"""
    w = _lwfa(60)
    with G.Sim(w.with_(particle_law="GT1", delta=0.45 * w.nzeta * w.h), bucket_capacity=40000) as s:
        s.step(8)
        assert not _two_ctas_per_sm(s) and s.diagnostics()["n_rejoined"] > 0
