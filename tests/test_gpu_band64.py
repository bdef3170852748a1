"""The band-limited evaluation of the FP64 path (csrc/band64.cuh) and of its
adjoint, the path against the oracle at sampled entries: the ends of its chirp and sample layouts, one chirp,
static and moving instances, time-division MIMO, no motion within a chirp, a mesh
lit from both sides (every chirp kept), targets too near or too fast for the
tables, few and many facets.

Tolerance: the phase of a path of some 60 m is 1e5 radians, so that FP64 rounding
alone leaves a few 1e-11 on either side; the interpolation adds 1e-13.  1e-9, as
for the direct sum; a wrong node, weight or reference shows at 1e-3.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2208_10939_gb300 as pkg
from paper_2208_10939_gb300 import autograd as bag
import scenegen as sg

pytestmark = pytest.mark.gpu

TOL = 1e-9


@pytest.fixture(scope="module")
def sim():
    s = pkg.Simulator(0)
    yield s
    s.close()


def check(sim, sc, n=200):
    sim.load_scene(sc)
    got = sim.simulate(pkg.PATH_FP64).cpu().numpy()
    r = sc.radar
    rng = np.random.default_rng(7)
    e = np.stack([rng.integers(0, r.O, n), rng.integers(0, r.N, n), rng.integers(0, r.M, n)], 1)
    ref = oracle.Frame(sc).adc_entries(e)
    err = np.linalg.norm(got[e[:, 0], e[:, 1], e[:, 2]] - ref) / np.linalg.norm(ref)
    assert err <= TOL, err


@pytest.mark.parametrize("M,N", [(32, 1), (64, 9), (96, 10), (128, 33), (224, 17), (256, 70),
                                 (544, 3), (1024, 19)])
def test_rows_and_chirps(sim, M, N):
    check(sim, sg.car_scene(seed=5, ntri=1200, M=M, N=N, P=2, Q=2, slant=24.0, speed=9.0))


@pytest.mark.parametrize("speed,N", [(0.0, 16), (0.3, 100), (15.0, 300), (300.0, 64)])
@pytest.mark.parametrize("tdm,intra", [(False, True), (True, True), (True, False)])
def test_motion(sim, speed, N, tdm, intra):
    sc = sg.car_scene(seed=6, ntri=600, M=128, N=N, P=2, Q=1, slant=22.0)
    sc.instances[0].vel = np.array([0.6 * speed, -0.8 * speed, 0.0])
    sc.radar.tdm = tdm
    sc.radar.intra_chirp_motion = intra
    check(sim, sc)


@pytest.mark.parametrize("two_sided", [False, True])
def test_instances(sim, two_sided):
    sc = sg.intersection_scene(seed=8, n_vehicles=3, M=256, N=24, P=2, Q=2, ground_n=16,
                               tri_scale=0.01)
    sc.instances[1].vel = np.zeros(3)
    sc.meshes[sc.instances[2].mesh_id].two_sided = two_sided
    check(sim, sc)


@pytest.mark.parametrize("y", [0.6, 3.0])
def test_near_plate(sim, y):
    """A plate nearer than its bounds allow, and one just beyond."""
    sc = sg.Scene([sg.plate(0.5, 0.5, 12)], [sg.Instance(0, np.array([0.1, y, 0.0]), np.eye(3),
                                                         np.array([0.0, 3.0, 0.0]))],
                  sg.make_radar(64, 12, 1, 2, 5.12e6, 30e12, 2.0, centre=(0.0, 0.0, 0.0)))
    check(sim, sc)


def _plate(n, size, vel, two_sided=False):
    m = sg.plate(size, size, n)
    m.two_sided = two_sided
    a = 0.3
    rot = np.array([[np.cos(a), -np.sin(a), 0.0], [np.sin(a), np.cos(a), 0.0], [0.0, 0.0, 1.0]])
    return sg.Scene([m], [sg.Instance(0, np.array([0.4, 9.0, 0.2]), rot, np.array(vel))],
                    sg.make_radar(96, 14, 1, 3, 5.12e6, 20e12, 2.0, centre=(0.0, 0.0, 0.0)))


def _car(speed, N, tdm=False, intra=True):
    sc = sg.car_scene(seed=6, ntri=500, M=128, N=N, P=2, Q=1, slant=22.0)
    sc.instances[0].vel = np.array([0.6 * speed, -0.8 * speed, 0.0])
    sc.radar.tdm = tdm
    sc.radar.intra_chirp_motion = intra
    return sc


# vertex, edge and series forms; static, all layouts, every chirp kept, every sample kept
ADJOINT = {"car": lambda: _car(9.0, 40), "static": lambda: _car(0.0, 9, tdm=True),
           "fast": lambda: _car(300.0, 12), "stepped": lambda: _car(9.0, 33, True, False),
           "edges": lambda: _plate(2, 0.6, [0.0, 2.0, 0.0]),
           "series": lambda: _plate(60, 0.02, [1.0, -3.0, 0.0]),
           "two_sided": lambda: _plate(4, 0.5, [0.5, 2.0, 0.0], True)}


@pytest.mark.parametrize("name", list(ADJOINT))
def test_adjoint(sim, name):
    """The cube is linear in the reflectivities: sum rho dL/drho = L, to the
    rounding of the paths.  A shift of all vertices against central
    differences of the cube: step 1e-6 m, (2 k h)^2 / 6 = 2e-6 of the largest
    derivative the loss can have, 2 k |W| |x|."""
    sc = ADJOINT[name]()
    es = bag.EchoScene(sim, sc)
    verts = es.vertex_tensor(sc, "cuda").requires_grad_(True)
    rho = torch.from_numpy(sc.meshes[0].rho.copy()).cuda().requires_grad_(True)
    adc = bag.echo(verts, rho, es)
    rng = np.random.default_rng(3)
    W = torch.from_numpy(rng.normal(size=adc.shape) + 1j * rng.normal(size=adc.shape)).cuda()
    loss = (W.conj() * adc).real.sum()
    loss.backward()
    scale = float(W.norm() * adc.detach().norm())
    lin = float((rho.detach().double() * rho.grad.double()).sum())
    # (the reflectivities' gradient is returned in their own float32)
    assert abs(lin - float(loss)) <= 1e-9 * scale + 2.0 ** -24 * float(
        (rho.detach() * rho.grad).abs().double().sum())
    h = 1e-6
    k = 2.0 * np.pi * (sc.radar.f0 + sc.radar.slope * sc.radar.M / sc.radar.fs) / 299792458.0
    for d in ([0.0, 1.0, 0.0], [0.6, 0.0, 0.8]):
        step = torch.tensor(d, dtype=torch.float64, device="cuda")
        with torch.no_grad():
            up = (W.conj() * bag.echo(verts + h * step, rho, es)).real.sum()
            dn = (W.conj() * bag.echo(verts - h * step, rho, es)).real.sum()
        fd = float(up - dn) / (2.0 * h)
        assert abs(fd - float((verts.grad * step).sum())) <= 5e-6 * 2.0 * k * scale
