"""The rate groups of the double-bounce synthesis (csrc/bounce.cuh) against the
FP64 path, which evaluates every chirp: row lengths below, at and beyond the
interpolation's 64-sample tiles, chirp counts from the first layout on,
time-division MIMO, slow and fast targets, more virtual facets of one rate than
a work item holds.

Tolerance: the double-bounce part's own bar, 1e-4 (FP32 records); a wrong
group, node, weight or reference shows at 1e-2.
"""
import numpy as np
import pytest
import torch

import paper_2208_10939_gb300 as pkg
import scenegen as sg

pytestmark = pytest.mark.gpu

TOL = 1e-4


@pytest.fixture(scope="module")
def sim():
    s = pkg.Simulator(0)
    yield s
    s.close()


def part(sim, sc, path):
    """the double-bounce echo alone"""
    out = []
    for on in (True, False):
        sc.radar.double_bounce = on
        sim.load_scene(sc)
        out.append(sim.simulate(path).to(torch.complex128))
    return out[0] - out[1]


def grouped(sim, sc):
    """the frame is one whose virtual facets are grouped (bounce_groups_apply)"""
    r = sc.radar
    sim.load_scene(sc)
    V = sim.simulate(pkg.PATH_MIXED, stats=True)[1]["n_bounce_facets"]
    assert V * r.Q * (r.N - 10) * r.M >= 8e7, V


@pytest.mark.parametrize("M,N,P,Q,tdm,speed", [
    (32, 10, 1, 1, False, 10.0), (96, 33, 2, 2, True, 8.0), (128, 64, 1, 3, False, 25.0),
    (192, 100, 2, 1, True, 3.0), (256, 16, 1, 2, False, 60.0), (64, 200, 2, 2, True, 1.0),
    (64, 48, 1, 1, False, 0.0)])
def test_groups(sim, M, N, P, Q, tdm, speed):
    sc = sg.car_ground_scene(ntri=1200, ground_n=6, M=M, N=N, P=P, Q=Q)
    sc.radar.tdm = tdm
    sc.instances[0].vel = np.array([0.3 * speed, -0.95 * speed, 0.0])
    got, ref = part(sim, sc, pkg.PATH_MIXED), part(sim, sc, pkg.PATH_FP64)
    err = float((got - ref).norm() / ref.norm())
    print(f"{M} x {N}, {P * Q} channels, {speed} m/s: {err:.2e}")
    assert float(ref.norm()) > 0 and err <= TOL


@pytest.mark.parametrize("beside", [False, True])
@pytest.mark.parametrize("at", [0.15, 0.5, 0.8])
def test_two_sided_second_facets_edge_on(sim, at, beside):
    """An upright two-sided plate over the ground that passes the antennas'
    plane at the fraction `at` of the frame: the second facets' obliquity |o|
    has a kink there; alone, or beside a weak one-sided plate whose facets are
    grouped.  Cubes in complex128, so that the part's difference
    takes no rounding from the ground's own echo."""
    m = sg.plate(0.4, 0.4, 8)
    m.two_sided = True
    radar = sg.make_radar(256, 64, 1, 2, 5.12e6, 30e12, 2.0, centre=(0.0, 0.0, 1.5))
    upright = np.array([[0.0, -1.0, 0.0], [1.0, 0.0, 0.0], [0.0, 0.0, 1.0]])
    speed, T = 12.0, 63 * radar.Tc
    sc = sg.Scene([m, sg.ground(6.0, 24, centre=(0.0, 7.0))],
                  [sg.Instance(0, (-speed * T * at, 10.0, 0.6), upright, (speed, 0.0, 0.0)),
                   sg.Instance(1, (0.0, 0.0, 0.0), np.eye(3), (0.0, 0.0, 0.0))], radar)
    if beside:
        sc.meshes.append(sg.plate(0.6, 0.6, 30, rho=1e-3))
        sc.instances.append(sg.Instance(2, (1.0, 11.0, 0.6), np.eye(3), (0.0, -9.0, 0.0)))

    def bounce(path):
        out = []
        for on in (True, False):
            sc.radar.double_bounce = on
            sim.load_scene(sc)
            out.append(sim.simulate(path, dtype=torch.complex128))
        return out[0] - out[1]

    got, ref = bounce(pkg.PATH_MIXED), bounce(pkg.PATH_FP64)
    err = float((got - ref).norm() / ref.norm())
    print(f"edge-on at {at}: {err:.2e}")
    if beside:
        sc.radar.double_bounce = True
        grouped(sim, sc)
    assert float(ref.norm()) > 0 and err <= TOL


@pytest.mark.parametrize("M,N,P,Q,tdm,speed", [
    (32, 260, 1, 1, False, 10.0), (96, 65, 2, 2, True, 8.0), (128, 33, 1, 3, False, 25.0),
    (192, 100, 2, 1, True, 3.0), (512, 16, 1, 3, False, 60.0), (64, 200, 2, 2, True, 1.0),
    (64, 80, 1, 3, False, 0.0)])
def test_groups_of_many_facets(sim, M, N, P, Q, tdm, speed):
    """As above with some 10k virtual facets a TX: fewer are not grouped."""
    sc = sg.car_ground_scene(ntri=6000, ground_n=24, M=M, N=N, P=P, Q=Q)
    sc.radar.tdm = tdm
    sc.instances[0].vel = np.array([0.3 * speed, -0.95 * speed, 0.0])
    grouped(sim, sc)
    got, ref = part(sim, sc, pkg.PATH_MIXED), part(sim, sc, pkg.PATH_FP64)
    err = float((got - ref).norm() / ref.norm())
    print(f"{M} x {N}, {P * Q} channels, {speed} m/s: {err:.2e}")
    assert float(ref.norm()) > 0 and err <= TOL
