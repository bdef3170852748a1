"""The band-limited evaluation of the mixed path (csrc/band.cuh) against the
plain FP64 path (itself checked against the oracle), where its layouts can go
wrong: row lengths of every lane grouping, one chirp, odd chirp counts, the
ends of the chirp layouts, static and moving instances together, instances
too wide or too fast for the tables, time-division MIMO, batches, frame
graphs after a mesh update.

Tolerance: the interpolation leaves 2e-6 at the band's edge, a phasor's FP32
steps about 1e-6, which a facet's vertex sum amplifies at most twice (the pair
form); the panels here are rough, so that the facets' sum does not cancel.
2e-5 covers that ten times; a wrong node, tap or reference shows at 1e-2.
"""
import numpy as np
import pytest
import torch

import paper_2208_10939_gb300 as pkg
import scenegen as sg

pytestmark = pytest.mark.gpu

TOL = 2e-5


@pytest.fixture(scope="module")
def sim():
    s = pkg.Simulator(0)
    yield s
    s.close()


def rough(scene, seed=1, sigma=0.012):
    rng = np.random.default_rng(seed)
    for m in scene.meshes:
        m.verts += rng.normal(scale=sigma, size=m.verts.shape)
    return scene


def check(sim, t0=None):
    got = sim.simulate(pkg.PATH_MIXED, t0=t0)
    ref = sim.simulate(pkg.PATH_FP64, t0=t0)
    err = float((got.to(ref.dtype) - ref).norm() / ref.norm())
    assert err <= TOL, err


@pytest.mark.parametrize("M,N", [(32, 1), (64, 2), (96, 11), (128, 12), (160, 13), (192, 25),
                                 (256, 33), (288, 7), (384, 17), (544, 3), (992, 5), (1024, 19),
                                 (512, 128)])
def test_rows_and_chirps(sim, M, N):
    sim.load_scene(rough(sg.car_scene(seed=5, ntri=4000, M=M, N=N, P=2, Q=2, slant=24.0, speed=9.0)))
    check(sim)


@pytest.mark.parametrize("speed,N", [(0.0, 16), (0.3, 100), (15.0, 300), (40.0, 200), (300.0, 64)])
def test_speeds(sim, speed, N):
    """Static (one chirp) to far beyond the chirp layouts (every chirp kept)."""
    sc = rough(sg.car_scene(seed=6, ntri=2500, M=128, N=N, P=2, Q=1, slant=22.0))
    sc.instances[0].vel = np.array([0.6 * speed, -0.8 * speed, 0.0])
    sim.load_scene(sc)
    check(sim)


@pytest.mark.parametrize("tdm", [False, True])
def test_static_and_moving_instances(sim, tdm):
    """Ground (too wide for the sample layouts), a parked car, two moving;
    against the direct sum (eight samples per lane), whose arithmetic static
    instances of large facets keep -- with its FP32 weights, 2.4e-5 from FP64
    on these 2.5 m ground cells -- and which is within TOL on rough vehicles."""
    sc = rough(sg.intersection_scene(seed=8, n_vehicles=3, M=256, N=24, P=3, Q=2, ground_n=40,
                                     tri_scale=0.03))
    sc.instances[1].vel = np.zeros(3)
    sc.radar.tdm = tdm
    sim.load_scene(sc)
    got = sim.simulate(pkg.PATH_MIXED)
    pkg.bart_set_synth_layout(sim.ctx, 8, 0)
    try:
        ref = sim.simulate(pkg.PATH_MIXED)
    finally:
        pkg.bart_set_synth_layout(sim.ctx, 0, 0)
    assert float((got - ref).norm() / ref.norm()) <= TOL


def test_near_wide_instance_keeps_every_sample(sim):
    """A moving wall around the antenna: the box bounds do not hold there."""
    m = sg.plate(30.0, 6.0, 40)
    sc = rough(sg.car_scene(seed=9, ntri=200, M=128, N=20, P=1, Q=2))
    sim.load_scene(rough(sg.Scene([m], [sg.Instance(0, (0.0, 4.0, 6.0), np.eye(3), (0.0, -3.0, 0.0))],
                                  sc.radar)))
    check(sim)


def test_batch_and_graph_after_mesh_update(sim):
    """Plans are made on the device: a replayed graph follows new vertices."""
    scenes = [rough(sg.batch_scene(i, N=20, tri_max=6000), seed=i) for i in range(3)]
    sim.load_scenes(scenes)
    check(sim)
    sc = rough(sg.car_scene(seed=3, ntri=3000, N=24, P=2, Q=2))
    sim.load_scene(sc)
    out = sim.simulate(pkg.PATH_MIXED)
    pkg.bart_set_graph(sim.ctx, True)
    try:
        sim.simulate(pkg.PATH_MIXED, out=out)
        v = torch.from_numpy(sc.meshes[0].verts * np.array([1.3, 1.5, 0.8])).cuda()
        pkg.bart_mesh_update(sim.ctx, 0, v)
        sim.simulate(pkg.PATH_MIXED, out=out, t0=0.02)
        torch.cuda.synchronize()
    finally:
        pkg.bart_set_graph(sim.ctx, False)
    ref = sim.simulate(pkg.PATH_FP64, t0=0.02)
    assert float((out.to(ref.dtype) - ref).norm() / ref.norm()) <= TOL


def test_record_counts_are_of_every_chirp(sim):
    sc = rough(sg.car_scene(seed=4, ntri=2000, M=128, N=30, P=1, Q=2))
    sim.load_scene(sc)
    st = sim.simulate(pkg.PATH_MIXED, stats=True)[1]
    ref = sim.simulate(pkg.PATH_FP64, stats=True)[1]
    assert st["n_terms"] == ref["n_terms"] and st["n_lit_pairs"] == ref["n_lit_pairs"]
    total = st["n_vertex"] + st["n_series"] + st["n_edge"]
    assert total == st["n_lit_pairs"] * 30
    for k in ("n_vertex", "n_series", "n_edge"):       # FP32 against FP64 at the forms' limits
        assert abs(st[k] - ref[k]) <= 1e-3 * total


def edge_on(at, two_sided=True, N=64):
    """A level 0.5 m plate 12 m out that passes the antennas' height at the
    fraction `at` of the frame, so that every facet's obliquity passes 0 there."""
    m = sg.plate(0.5, 0.5, 4)
    m.two_sided = two_sided
    radar = sg.make_radar(128, N, 2, 2, 5.12e6, 30e12, 2.0, centre=(0.0, 0.0, 0.0))
    level = np.array([[1.0, 0.0, 0.0], [0.0, 0.0, -1.0], [0.0, 1.0, 0.0]])
    speed, T = 12.0, (N - 1) * radar.Tc
    return sg.Scene([m], [sg.Instance(0, (0.2, 12.0, -speed * T * at), level, (0.0, 0.0, speed))], radar)


@pytest.mark.parametrize("path", [pkg.PATH_MIXED, pkg.PATH_SPECTRAL])
@pytest.mark.parametrize("at", [0.1, 0.5, 0.93])
def test_two_sided_facets_edge_on(sim, path, at):
    """A two-sided facet's obliquity |o| has a kink where it passes edge-on,
    which no interpolation over the chirps follows.  The bar is the path's own,
    1e-4: a flat panel's facets cancel, which amplifies the records' FP32
    rounding; an interpolated kink leaves 1e-2."""
    sim.load_scene(edge_on(at))
    got, ref = sim.simulate(path), sim.simulate(pkg.PATH_FP64)
    err = float((got.to(ref.dtype) - ref).norm() / ref.norm())
    print(f"edge-on at {at}, path {path}: {err:.2e}")
    assert float(ref.norm()) > 0 and err <= 1e-4
