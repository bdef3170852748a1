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
