"""The two-kernel step of small contexts (wide.cu, the default there) against the general
kernels, which an explicit overlap option selects: same state after the same steps, at ring
sizes on the edges of its splits, in every scheme, storage and boundary it accepts, across
call boundaries and a change of path in mid-run. In single precision only long rings take
it (the short sizes then compare the general kernels with themselves)."""
import numpy as np
import pytest

import oracle as o
from paper_1903_03356_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# both paths round alike but for the order of sums (as fused against separate kernels)
AGREE = {"fp64": 1e-12, "fp32": 2e-6, "fp16": 2e-3}


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_03356_gb300 import lbmib
    return lbmib


def rings(sizes, ka=0.0, nx=203, ny=64, walls=True):
    """Circles of the given vertex counts side by side, between walls or in a periodic box."""
    caps, x = [], 16.0
    for k, n in enumerate(sizes):
        r = 1.5 if n < 8 else min(0.8 * n / (2.0 * np.pi), 12.0 if n < 256 else 20.0)
        xy = W.circle(n, r, x + r + 0.113, 30.07 + 1.3 * k)
        x += 2.0 * r + 4.0
        m = W.node_mass(1.0, W.signed_area(xy), n)
        caps.append(W.Capsule(xy, 0.01, W.kb_from_eb(W.stable_eb(0.01, 0.01, r, xy, m), 0.01, r), ka, m))
    return W.Case("rings", nx, ny, 0.7, walls, gx=W.poiseuille_force(0.7, 0.02, ny), init="parabola", capsules=caps)


def pair(L, case, storage, repulsion=0.0, **opts):
    out = []
    for general in (False, True):
        ctx = L.from_case(case, storage=storage)
        ctx.set_option(L.OPT_GRAPH_STEPS, 8)
        if repulsion:
            ctx.set_repulsion(repulsion)
        for k, v in opts.items():
            ctx.set_option(getattr(L, k), v)
        if general:
            ctx.set_option(L.OPT_OVERLAP, 0)
        out.append(ctx)
    return out


def agree(a, b, case, tol):
    np.testing.assert_allclose(a.read_populations(), b.read_populations(), rtol=0, atol=tol)
    for k in range(len(case.capsules)):
        xa, va = a.read_capsule(k)[:2]
        xb, vb = b.read_capsule(k)[:2]
        np.testing.assert_allclose(xa, xb, rtol=0, atol=10 * tol)
        np.testing.assert_allclose(va, vb, rtol=0, atol=10 * tol)
    np.testing.assert_allclose(a.observables_all(), b.observables_all(), rtol=1e3 * tol, atol=1e3 * tol)


@pytest.mark.parametrize("scheme", [o.KINEMATIC, o.DYNAMIC])
@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("sizes", [(3,), (16, 17), (127, 5, 33), (257, 6), (1024,)])
def test_ring_sizes(L, scheme, storage, sizes):
    case = rings(sizes)
    a, b = pair(L, case, storage)
    for ctx in (a, b):
        for n in (1, 8, 13):
            ctx.step(n, scheme)
    agree(a, b, case, AGREE[storage])


@pytest.mark.parametrize("scheme", [o.KINEMATIC, o.DYNAMIC])
@pytest.mark.parametrize("storage", ["fp64", "fp32"])
def test_area_force_periodic_box_and_direct_launches(L, scheme, storage):
    case = rings((300, 40), ka=0.05, walls=False)
    a, b = pair(L, case, storage, OPT_GRAPHS=0)
    for ctx in (a, b):
        ctx.step(21, scheme)
    agree(a, b, case, AGREE[storage])


@pytest.mark.parametrize("scheme", [o.KINEMATIC, o.DYNAMIC])
def test_repulsion_and_fp64_interpolation_over_fp32(L, scheme):
    case = W.dense_biconcave(nx=300, ny=150, count=6, n=200, hematocrit=0.3, seed=4, scheme=scheme)
    a, b = pair(L, case, "fp64", repulsion=2.0)
    for ctx in (a, b):
        ctx.step(19, scheme)
    agree(a, b, case, 1e-12)
    long_rings = W.dense_biconcave(nx=300, ny=150, count=6, n=300, hematocrit=0.3, seed=4, scheme=scheme)
    a, b = pair(L, long_rings, "fp32", repulsion=2.0)
    for ctx in (a, b):
        ctx.step(19, scheme)
    agree(a, b, long_rings, AGREE["fp32"])
    a, b = pair(L, case, "fp32", OPT_IB_FP64=1)
    for ctx in (a, b):
        ctx.step(19, scheme)
    agree(a, b, case, AGREE["fp32"])


@pytest.mark.parametrize("scheme", [o.KINEMATIC, o.DYNAMIC])
@pytest.mark.parametrize("storage", ["fp64", "fp32"])
def test_open_channel(L, scheme, storage):
    case = W.open_channel_capsule(ny=60, length=3.0, diameter=28.0, scheme=scheme)
    a, b = pair(L, case, storage)
    for ctx in (a, b):
        ctx.step(30, scheme)
    agree(a, b, case, AGREE[storage])


def test_paths_alternate_and_states_load(L):
    # the state between calls is the same whichever kernels made it: list, force field, history
    case = rings((64, 31))
    a, b = pair(L, case, "fp64")
    for n, general in ((5, False), (6, True), (9, False), (1, True), (12, False)):
        a.set_option(L.OPT_OVERLAP, 0 if general else -1)
        a.step(n, o.DYNAMIC if n % 2 else o.KINEMATIC)
        b.step(n, o.DYNAMIC if n % 2 else o.KINEMATIC)
    agree(a, b, case, 1e-12)
    np.testing.assert_allclose(a.read_force_field(), b.read_force_field(), rtol=0, atol=1e-14)
    c = L.from_case(case, storage="fp64")
    c.load_state(a.save_state())
    for ctx in (a, b, c):
        ctx.step(11, o.DYNAMIC)
    agree(c, b, case, 1e-12)


@pytest.mark.parametrize("scheme", [o.KINEMATIC, o.DYNAMIC])
@pytest.mark.parametrize("general", [False, True])
def test_repeated_rests_of_calls(L, scheme, general):
    # calls that leave the same number of steps over replay a captured rest; others do not
    case = rings((64, 31))
    a, b = pair(L, case, "fp64", OPT_OVERLAP=1 if general else -1)
    if not general:
        b.set_option(L.OPT_OVERLAP, -1)
    b.set_option(L.OPT_GRAPHS, 0)
    n0 = a.launch_count, b.launch_count
    for n in (5, 5, 5, 7, 5, 11, 11, 11, 1, 1, 4):
        a.step(n, scheme)
        b.step(n, scheme)
    agree(a, b, case, 1e-12)
    assert a.launch_count - n0[0] >= b.launch_count - n0[1]   # graphs of 8 close and open their own spreads


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("nx, ny", [(3, 5), (5, 40), (259, 33), (1027, 301)])
def test_ragged_lattices(L, storage, nx, ny):
    # rows that no vector fits: one thread per node below 2^18 nodes, beside the vector kernel above
    case = W.Case("ragged", nx, ny, 0.7, True, -0.02, 0.02, gx=1e-5, init="shear")
    ctx = L.from_case(case, storage=storage)
    ctx.step(9, o.KINEMATIC)
    s = o.Sim(o.lattice(nx, ny, 0.7, True, -0.02, 0.02, 1e-5, 0.0))
    s.init_fields(*case.fields())
    s.step(9, o.KINEMATIC)
    tol = {"fp64": 1e-15, "fp32": 5e-9, "fp16": 1e-4}[storage]   # rounding of nine steps of |f - w| < 1e-2
    np.testing.assert_allclose(ctx.read_populations(), s.populations(), rtol=0, atol=tol)


def test_support_error_is_reported(L):
    case = rings((64,))
    ctx = L.from_case(case, storage="fp32")
    ctx.set_capsule_positions(0, case.capsules[0].xy - np.array([0.0, 25.0]))
    ctx.step(3, o.DYNAMIC)
    with pytest.raises(L.LbmibError) as e:
        ctx.sync()
    assert e.value.status == L.ERR_SUPPORT
