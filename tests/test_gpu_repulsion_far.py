"""The repulsion's float tests where rounding matters: rings that have drifted millions of
periods through the periodic axes, and pairs within 1e-5 of the cut-off across the seam,
against the FP64 oracle."""
import numpy as np
import pytest

import oracle as o
from paper_1903_03356_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_03356_gb300 import lbmib
    return lbmib


def ring(n, r, cx, cy, phase=0.137):
    t = 2 * np.pi * (np.arange(n) + phase) / n
    return np.stack([cx + r * np.cos(t), cy + r * np.sin(t)], axis=1)


def pair(xys, nx=80, ny=40, walls=False):
    caps = [W.Capsule(xy, 0.02, 0.002, 0.0, W.node_mass(1.0, W.signed_area(xy), len(xy))) for xy in xys]
    return W.Case("pair", nx, ny, 0.8, walls, gx=1e-6, init="rest", capsules=caps)


def oracle_run(case, scheme, rc, steps, coeff=o.REPULSION_COEFF):
    s = o.Sim(o.lattice(case.nx, case.ny, case.tau, case.walls, 0.0, 0.0, case.gx, case.gy))
    s.init_fields(*case.fields())
    for c in case.capsules:
        s.add_capsule(c.xy, c.ks, c.kb, c.ka, c.mass)
    s.set_repulsion(rc, coeff)
    assert s.step(steps, scheme) == 0
    return s


@pytest.mark.parametrize("scheme", [o.KINEMATIC, o.DYNAMIC])
@pytest.mark.parametrize("periods", [(300, -300), (312_500, 0), (-1_562_509, 3_906_251), (2_812_500, 0)])
def test_rings_far_from_the_origin(L, scheme, periods):
    # up to 9e8 nodes, where floats are 64 apart: these rings' coarse cells of 36 x 43 nodes would
    # come out two apart. The coefficient makes a step's force move a vertex by about 1e-3.
    coeff, steps = 5e-3, 4
    case = pair([ring(48, 7.0, 88.3, 60.07), ring(48, 7.0, 103.1, 60.57)], 320, 128)
    s = oracle_run(case, scheme, 2.0, steps, coeff)
    off = oracle_run(case, scheme, 2.0, steps, 1e-30)
    effect = np.abs(s.read_capsule(0)[0] - off.read_capsule(0)[0]).max()
    for far in ((0, 1), (1,)):     # both rings, and one while the other stays at home
        ctx = L.from_case(case, storage="fp64")
        ctx.set_repulsion(2.0, coeff)
        shift = np.zeros((2, 2))
        for k in far:
            shift[k] = 320.0 * periods[0], 128.0 * periods[1]
            ctx.set_capsule_positions(k, case.capsules[k].xy + shift[k])
        ctx.step(steps, scheme)
        ctx.sync()
        # the start and each step round a position by half a place, and with it the distances
        # (of 0.9, d^-2.5: four times their rounding of the step's 1e-3), velocities and strains
        tol = 1e-10 + 4 * (steps + 1) * np.spacing(float(np.abs(shift).max()))
        assert effect > 20.0 * tol
        for k in range(2):
            np.testing.assert_allclose(ctx.read_capsule(k)[0].reshape(-1, 2) - shift[k],
                                       s.read_capsule(k)[0].reshape(-1, 2), rtol=0, atol=tol)


@pytest.mark.parametrize("axis", ["x", "y"])
@pytest.mark.parametrize("off", [-1e-5, 1e-5])
def test_pairs_at_the_cut_off_across_the_seam(L, axis, off):
    # two rings whose nearest vertices face each other over the periodic seam, r_c + off apart
    rc, r, n = 2.0, 7.0, 48
    gap = rc + off
    if axis == "x":
        xys = [ring(n, r, 72.3, 20.07, 0.0), ring(n, r, 72.3 + 2 * r + gap - 80.0, 20.07, 0.0)]
    else:
        xys = [ring(n, r, 40.3, 32.07, 0.0), ring(n, r, 40.3, 32.07 + 2 * r + gap - 40.0, 0.0)]
    case = pair(xys)
    s = oracle_run(case, o.DYNAMIC, rc, 1)
    ctx = L.from_case(case, storage="fp64")
    ctx.set_repulsion(rc)
    ctx.step(1, o.DYNAMIC)
    ctx.sync()
    for k in range(2):
        np.testing.assert_allclose(ctx.read_capsule(k)[0], s.read_capsule(k)[0], rtol=0, atol=1e-12)
    # one pair's force moves a vertex by far more than that
    coeff = 1e-4 / (8.0 * np.sqrt(2.0))
    assert 0.5 * coeff * rc ** -2.5 / case.capsules[0].mass > 1e-8
