"""The spectral kernel (csrc/spectral.cu) against the oracle on the frames that
it serves: the other delay forms, frames longer than the band-limited
evaluation's tables, many tiny instances -- with thousands of facets, so that
its record queues, the spreading of neighbouring lines and the edge and series
records over many facets are all in use.

Bar: the path's own, 1e-4 relative L2.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2208_10939_gb300 as pkg
import scenegen as sg

pytestmark = pytest.mark.gpu

TOL = 1e-4


@pytest.fixture(scope="module")
def sim():
    s = pkg.Simulator(0)
    yield s
    s.close()


def check(got, sc):
    ref = oracle.Frame(sc).adc_full()
    err = float(np.linalg.norm(got.cpu().numpy() - ref) / np.linalg.norm(ref))
    print(f"{sc.name} M={sc.radar.M} N={sc.radar.N}: {err:.2e}")
    assert err <= TOL


def car(form, ntri=4000, M=256, N=4, tdm=False, seed=5, **kw):
    sc = sg.car_scene(seed=seed, ntri=ntri, M=M, N=N, P=2, Q=2, slant=24.0, **kw)
    sc.radar.tdm = tdm
    setattr(sc.radar, form, True)
    return sc


@pytest.mark.parametrize("form", ["delay_ref", "far_field"])
@pytest.mark.parametrize("M,N,tdm", [(32, 3, False), (96, 4, True), (256, 5, False), (768, 2, True),
                                     (1024, 2, False)])
def test_delay_forms(sim, form, M, N, tdm):
    sc = car(form, M=M, N=N, tdm=tdm)
    sim.load_scene(sc)
    check(sim.simulate(pkg.PATH_SPECTRAL), sc)


@pytest.mark.parametrize("form", ["delay_ref", "far_field"])
def test_record_forms(sim, form):
    """A coarse ground's vertex and edge records, the series records of a fine plate
    seen at a right angle."""
    sc = car(form, ntri=1500, M=128, N=3)
    sc.meshes += [sg.ground(12.0, 12, centre=(2.0, 20.0)), sg.plate(0.2, 0.2, 40)]
    sc.instances += [sg.Instance(1, (0.0, 0.0, 0.0), np.eye(3), (0.0, 0.0, 0.0)),
                     sg.Instance(2, (0.0, 14.0, 6.0), np.eye(3), (1.0, -6.0, 0.0))]
    sim.load_scene(sc)
    got, st = sim.simulate(pkg.PATH_SPECTRAL, stats=True)
    assert min(st["n_vertex"], st["n_series"], st["n_edge"]) > 0
    check(got, sc)


def test_long_frame(sim):
    sc = sg.car_scene(seed=5, ntri=900, M=32, N=1025, P=1, Q=1, slant=22.0)
    sim.load_scene(sc)
    check(sim.simulate(pkg.PATH_SPECTRAL), sc)


def test_many_tiny_instances(sim):
    rng = np.random.default_rng(2)
    ins = [sg.Instance(0, (rng.uniform(-8, 8), rng.uniform(10, 35), rng.uniform(0, 3)),
                       sg.rot_z(rng.uniform(-0.3, 0.3)), (0.0, rng.uniform(-10, 10), 0.0))
           for _ in range(64)]
    sc = sg.Scene([sg.plate(0.2, 0.2, 3)], ins, sg.make_radar(128, 6, 2, 2, 5.12e6, 12.5e12, 2.0),
                  name="plates")
    sim.load_scene(sc)
    check(sim.simulate(pkg.PATH_SPECTRAL), sc)


def test_batch(sim):
    scenes = [car("delay_ref", ntri=n, M=128, N=3, seed=k) for k, n in enumerate((2500, 600, 1200))]
    sim.load_scenes(scenes)
    got = sim.simulate(pkg.PATH_SPECTRAL)
    for b, sc in enumerate(scenes):
        check(got[b], sc)


@pytest.mark.parametrize("form", ["delay_ref", "far_field"])
@pytest.mark.parametrize("M", [96, 128])
def test_lines_beyond_a_cycle_per_sample(sim, form, M):
    """Vertices up to 9 m from their facet's centroid under a steep, slowly
    sampled chirp: lines two cycles per sample from it, whose cells are those of
    the alias.  The FP32 line rate leaves 2^-23 x M / 2 cycles, 2e-5 rad at most,
    and facets this large have no cancelling weights: the path's bar."""
    radar = sg.make_radar(M, 3, 1, 2, 2e6, 80e12, 2.0, centre=(0.0, 0.0, 2.0))
    setattr(radar, form, True)
    a = np.deg2rad(50.0)
    tilt = np.array([[1.0, 0.0, 0.0], [0.0, np.cos(a), -np.sin(a)], [0.0, np.sin(a), np.cos(a)]])
    sc = sg.Scene([sg.plate(9.0, 24.0, 2)],
                  [sg.Instance(0, (3.0, 60.0, 1.0), sg.rot_z(0.2) @ tilt, (0.5, -4.0, 0.0))], radar,
                  name="panel")
    c = sc.meshes[0].verts[sc.meshes[0].tris] @ sc.instances[0].rot.T
    u = 2.0 * (c - c.mean(1, keepdims=True))[..., 1]           # about along the line of sight
    assert np.abs(u).max() * radar.slope / (radar.fs * 299792458.0) > 1.2
    sim.load_scene(sc)
    check(sim.simulate(pkg.PATH_SPECTRAL), sc)
