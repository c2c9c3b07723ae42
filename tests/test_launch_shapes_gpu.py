"""Launch shapes a call of s-steps chooses from: the same s-steps must come out of each of them.

2-D marches whose particles are shared by 1, 2, 4 or 8 CTAs against the one-CTA march
(cluster_ctas = 1 allows no other), over the options of the 2-D path; 128 x 128 FP32 marches with
two CTAs per SM (many s-steps per call) against one s-step per call.  FP32 transverse currents
add in fixed point, so the FP32 states are equal bit for bit.  Stored particles deposit by float
reductions in global memory, whose order several CTAs do not fix: those options are compared
in FP64, to rounding (in FP32 a GT1 run's stops amplify the last bit by 10^3 per s-step)."""
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


OPTIONS = {
    "plain": {}, "channel": dict(channel=W.Channel(0.25, 20.0)),
    "refined": dict(hz=True), "trapping": dict(delta=3.0), "gt1": dict(particle_law="GT1", delta=8.0),
    "snapshot": dict(snapshot=True, capture_current=True),
    "beam": dict(beam=W.Beam(n_peak=0.002, sigma_r=3.0, sigma_z=1.5, zeta_center=8.0, gamma=200.0,
                             n_macro=500)),
}


@pytest.mark.parametrize("option", list(OPTIONS))
@pytest.mark.parametrize("precision,nx,ppc", [(64, 64, 3), (64, 128, 4), (32, 32, 5), (32, 128, 4),
                                              (32, 512, 2), (32, 1024, 1)])
def test_2d_shapes_equal_one_cta(G, option, precision, nx, ppc):
    if precision == 32 and option in ("trapping", "gt1", "beam"):
        pytest.skip("compared in FP64")
    w = W.small_2d(nx=nx, nzeta=50, ppc=ppc, precision=precision, a0=2.0, delta=20.0)
    kw = dict(OPTIONS[option])
    if kw.pop("hz", False):
        kw["hz"] = W.refined_h(w.nzeta, w.h, 2.0)
    w = w.with_(**kw)
    stored = option in ("trapping", "gt1", "beam")
    tol = 1e-11 if precision == 64 else 0.0
    cap = {"bucket_capacity": 4096} if stored else {}
    with G.Sim(w, cluster_ctas=1, **cap) as a, G.Sim(w, **cap) as b, G.Sim(w, **cap) as c:
        for n in (1, 2, 5):                          # different shapes as n grows
            a.step(n)
            b.step(n)
            for _ in range(n):
                c.step(1)                            # the widest split
            ra = a.state()
            for v in (b, c):
                rv = v.state()
                for comp in range(6):
                    scale = np.abs(ra[:4] if comp < 4 else ra[4:]).max()
                    assert np.abs(rv[comp] - ra[comp]).max() <= tol * scale, (n, comp)
                da, dv = a.diagnostics(), v.diagnostics()
                for k in ("n_trapped", "n_stored", "n_rejoined", "pushes", "step"):
                    assert da[k] == dv[k], (n, k, da[k], dv[k])
                for k in ("field_energy", "kinetic_energy", "charge_flux", "stored_kinetic_energy"):
                    assert abs(da[k] - dv[k]) <= max(tol, 1e-5 if precision == 32 else 1e-12) * abs(da[k]) + 1e-30, k
                assert np.abs(a.onaxis_ez() - v.onaxis_ez()).max() <= tol * np.abs(a.onaxis_ez()).max()
            if option == "snapshot":
                # (B_z of an x-polarised 2-D run is zero: fields are compared on E_x's scale)
                for f, of in (("Ex", "Ex"), ("Bz", "Ex"), ("jx", "jx"), ("jz", "jx")):
                    x, y = a.fields(f), c.fields(f)
                    assert np.abs(x - y).max() <= tol * np.abs(a.fields(of)).max()
                assert np.abs(a.current() - c.current()).max() <= tol * np.abs(a.current()).max()


@pytest.mark.parametrize("nz,ppc,a0,n", [(120, 2, 1.0, 16), (96, 1, 1.5, 17), (90, 5, 1.0, 14),
                                           (300, 1, 1.0, 19)])
def test_128_two_ctas_per_sm_equal_single_steps(G, nz, ppc, a0, n):
    """More s-steps than one CTA per SM keeps in flight: marches with two CTAs per SM."""
    w = W.lwfa_3d_128x128x1024()
    w = w.with_(nzeta=nz, species=[W.Species(-1.0, 1.0, w.species[0].density, ppc)],
                laser=W.Laser(**{**w.laser.__dict__, "a0": a0, "zeta_center": 0.5 * nz * w.h}))
    with G.Sim(w) as a, G.Sim(w) as b:
        assert a.launch_shape()["pipeline"] < n
        a.step(n)
        for _ in range(n):
            b.step(1)
        assert np.array_equal(a.state(), b.state())
        da, db = a.diagnostics(), b.diagnostics()
        for k in ("n_trapped", "n_stored", "n_rejoined", "pushes", "step"):
            assert da[k] == db[k]
        for k in ("field_energy", "kinetic_energy", "charge_flux"):
            assert abs(da[k] - db[k]) <= 1e-5 * abs(db[k])
        assert np.array_equal(a.onaxis_ez(), b.onaxis_ez())


def test_128_two_ctas_per_sm_with_a_beam(G):
    """Stored particles (pushed along s, depositing, rejoining) in marches with two CTAs per SM."""
    w = W.pwfa_3d_128x128x768(n_macro=1 << 14)
    w = w.with_(nzeta=90, beam=W.Beam(**{**w.beam.__dict__, "n_peak": 0.05, "zeta_center": 45 * w.h,
                                         "sigma_z": 0.2}))
    with G.Sim(w) as a, G.Sim(w) as b:
        a.step(14)
        for _ in range(14):
            b.step(1)
        sa, sb = a.state(), b.state()
        assert np.abs(sa - sb).max() <= 1e-3 * np.abs(sb).max()
        da, db = a.diagnostics(), b.diagnostics()
        assert da["n_stored"] == db["n_stored"] > 0 and da["pushes"] == db["pushes"]
        assert abs(da["field_energy"] - db["field_energy"]) <= 1e-3 * db["field_energy"]


@pytest.mark.parametrize("nz,n", [(640, 14), (637, 9), (640, 7)])
def test_128_streamed_equal_single_steps(G, nz, n):
    """Streamed calls that march with two CTAs per SM (and 7 s-steps, which do not, from pageable
    memory); a ragged last group of slices."""
    import torch
    w = W.lwfa_3d_128x128x1024()
    w = w.with_(nzeta=nz, laser=W.Laser(**{**w.laser.__dict__, "zeta_center": 0.5 * nz * w.h}))
    with G.Sim(w) as a, G.Sim(w) as b:
        host = a.state()
        if n != 7:
            pinned = torch.empty(host.shape, dtype=torch.complex64, pin_memory=True).numpy()
            pinned[...] = host
            host = pinned
        diags = a.step_streamed(n, host)
        for i in range(n):
            b.step(1)
            assert diags[i]["pushes"] == b.diagnostics()["pushes"]
        assert np.array_equal(host, b.state())
        assert np.array_equal(a.state(), host)
        assert np.array_equal(a.onaxis_ez(), b.onaxis_ez())
