"""Which kernels a step takes, by their number: the two-kernel step launches 2n + 1 kernels for
n steps enqueued directly, the general kernels 3n + 1 (one CTA per capsule, update and next
spread fused) or 4n; and that a context that keeps the general kernels computes what it does
with them asked for by name."""
import numpy as np
import pytest

import oracle as o
from paper_1903_03356_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N = 6


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_03356_gb300 import lbmib
    return lbmib


def rows(count, n, nx, ny, radius):
    """`count` circles of n vertices in rows between walls."""
    cols = int(nx // (2.0 * radius + 6.0))
    caps = []
    for k in range(count):
        xy = W.circle(n, radius, (k % cols + 0.5) * nx / cols + 0.0137, 5.0 + radius + (k // cols) * (2.0 * radius + 5.0))
        caps.append(W.Capsule(xy, 0.01, 0.001, 0.0, W.node_mass(1.0, W.signed_area(xy), n)))
        assert xy[:, 1].max() < ny - 4.0
    return W.Case("rows", nx, ny, 0.8, True, -0.005, 0.005, gx=1e-7, init="shear", capsules=caps)


def launches(L, case, storage, scheme, **opts):
    """Kernels of N steps enqueued directly."""
    ctx = L.from_case(case, storage=storage)
    ctx.set_option(L.OPT_GRAPHS, 0)
    for k, v in opts.items():
        ctx.set_option(getattr(L, k), v)
    n0 = ctx.launch_count
    ctx.step(N, scheme)
    count = ctx.launch_count - n0
    ctx.sync()
    ctx.close()
    return count


TWO, FUSED, SPLIT = 2 * N + 1, 3 * N + 1, 4 * N


@pytest.mark.parametrize("scheme", [o.KINEMATIC, o.DYNAMIC])
@pytest.mark.parametrize("count, n, nx, ny, radius", [(1, 300, 160, 120, 30.0), (60, 128, 900, 500, 16.0)])
@pytest.mark.parametrize("ib_fp64", [0, 1])
def test_fp16_storage_keeps_the_general_kernels(L, scheme, count, n, nx, ny, radius, ib_fp64):
    case = rows(count, n, nx, ny, radius)
    assert launches(L, case, "fp16", scheme, OPT_IB_FP64=ib_fp64) == SPLIT


def test_fp16_results_are_those_of_the_general_kernels(L):
    # FP64 interpolations: the general kernels then add their shares in double and repeat
    # themselves; a share rounded differently at every node parts FP16 populations by 1e-4
    case = rows(60, 128, 900, 500, 16.0)
    out = []
    for overlap in (-1, 1):
        ctx = L.from_case(case, storage="fp16")
        ctx.set_option(L.OPT_IB_FP64, 1)
        ctx.set_option(L.OPT_OVERLAP, overlap)
        ctx.step(40, o.DYNAMIC)
        ctx.sync()
        out.append(ctx.field_view(L.FIELD_POPULATIONS)[:, :, :case.nx].double().cpu().numpy())   # less the rest weights
    assert np.linalg.norm(out[0] - out[1]) < 1e-5 * np.linalg.norm(out[1])


@pytest.mark.parametrize("scheme", [o.KINEMATIC, o.DYNAMIC])
def test_fp16_runs_part_by_few_storage_steps(L, scheme):
    # the order of the tiles' float additions is free: two runs, and the schedules with and
    # without the overlap, may part by storage steps (2^-11) in a hundredth of the populations
    case = W.poiseuille_biconcave(2048, 1024, count=256, n=128, a=8.0, seed=3, scheme=scheme, placement="grid")
    out = []
    for overlap in (-1, -1, 0):
        ctx = L.from_case(case, storage="fp16")
        ctx.set_option(L.OPT_OVERLAP, overlap)
        ctx.step(50, scheme)
        ctx.sync()
        out.append(ctx.field_view(L.FIELD_POPULATIONS)[:, :, :case.nx].float().cpu().numpy())
    for other in out[1:]:
        assert np.linalg.norm(other - out[0]) < 2.0 ** -11 / np.sqrt(100.0) * np.linalg.norm(out[0])


# (count, n, nx, ny, radius): CTAs with a multiprocessor each (up to 120) and beyond, vertices
# closer than 0.65 nodes and (the names with "far") farther apart
SIZES = {"8x256": (8, 256, 500, 160, 15.0), "8x384": (8, 384, 500, 160, 20.0), "8x400": (8, 400, 500, 160, 20.0),
         "8x384 far": (8, 384, 500, 260, 45.0), "8x400 far": (8, 400, 500, 260, 45.0),
         "1x384": (1, 384, 120, 80, 25.0), "1x392": (1, 392, 120, 80, 25.0),
         "2x512": (2, 512, 240, 100, 30.0), "2x512 far": (2, 512, 320, 170, 70.0),
         "2x776": (2, 776, 240, 100, 30.0), "2x808 far": (2, 808, 500, 250, 100.0),
         "15x400": (15, 400, 700, 200, 20.0), "16x384": (16, 384, 700, 200, 20.0), "16x400": (16, 400, 700, 200, 20.0),
         "16x192": (16, 192, 700, 200, 15.0), "16x200": (16, 200, 700, 200, 15.0),
         "16x256 far": (16, 256, 700, 400, 35.0), "16x264 far": (16, 264, 700, 400, 35.0),
         "16x128": (16, 128, 700, 200, 20.0), "64x128": (64, 128, 600, 300, 12.0)}


@pytest.mark.parametrize("storage, ib_fp64, scheme, general", [
    ("fp64", 0, o.DYNAMIC, {"8x400", "1x392", "2x512", "2x776", "15x400", "16x384", "16x400", "16x200", "16x264 far", "64x128"}),
    ("fp64", 0, o.KINEMATIC, {"2x776", "16x400"}),
    ("fp32", 1, o.DYNAMIC, set(SIZES) - {"8x256", "8x384 far", "16x128"}),
    ("fp32", 1, o.KINEMATIC, set(SIZES) - {"8x256", "8x384", "1x384", "8x384 far", "8x400 far", "2x512 far", "16x128"})])
def test_two_kernel_lines_with_fp64_interpolations(L, storage, ib_fp64, scheme, general):
    for name, size in SIZES.items():
        count = launches(L, rows(*size), storage, scheme, OPT_IB_FP64=ib_fp64)
        assert (count != TWO) == (name in general), (name, count)


@pytest.mark.parametrize("scheme", [o.KINEMATIC, o.DYNAMIC])
@pytest.mark.parametrize("size", ["2x512 far", "8x384", "16x256 far"])
def test_fp64_ctas_alone_and_shared_against_the_general_kernels(L, scheme, size):
    case = rows(*SIZES[size])
    a, b = L.from_case(case, storage="fp64"), L.from_case(case, storage="fp64")
    b.set_option(L.OPT_OVERLAP, 1)
    for ctx in (a, b):
        ctx.step(12, scheme)
    np.testing.assert_allclose(a.read_populations(), b.read_populations(), rtol=0, atol=1e-12)
    for k in range(len(case.capsules)):
        np.testing.assert_allclose(a.read_capsule(k)[0], b.read_capsule(k)[0], rtol=0, atol=1e-11)


@pytest.mark.parametrize("scheme", [o.KINEMATIC, o.DYNAMIC])
def test_two_kernel_lines_in_single_precision(L, scheme):
    for size, count in {(1, 256, 160, 120, 30.0): SPLIT, (1, 257, 160, 120, 30.0): TWO,
                        (60, 64, 700, 300, 10.0): SPLIT, (60, 65, 700, 300, 10.0): TWO,
                        (152, 33, 700, 300, 6.0): TWO, (152, 32, 700, 300, 6.0): FUSED,
                        (153, 33, 700, 300, 6.0): FUSED, (400, 64, 900, 700, 10.0): FUSED,
                        (2, 300, 1024, 1024, 30.0): TWO, (2, 300, 1024, 1025, 30.0): SPLIT,
                        # vertices closer than 0.45 nodes, on shared multiprocessors and alone
                        (16, 384, 700, 200, 20.0): SPLIT, (15, 384, 700, 200, 20.0): TWO,
                        (64, 128, 600, 300, 8.0): TWO if scheme == o.KINEMATIC else SPLIT,
                        (64, 132, 600, 300, 8.0): SPLIT}.items():
        assert launches(L, rows(*size), "fp32", scheme) == count, size


def test_changing_leftovers_are_captured_a_few_times_only(L):
    case = rows(2, 40, 200, 60, 8.0)
    a, b = L.from_case(case, storage="fp64"), L.from_case(case, storage="fp64")
    b.set_option(L.OPT_GRAPHS, 0)

    def go(*lengths):
        before = a.capture_count
        for n in lengths:
            a.step(n, o.DYNAMIC)
            b.step(n, o.DYNAMIC)
        return a.capture_count - before

    assert go(4, 6, 4, 6, 1, 1, 1) == 0        # no length twice in a row, and single steps
    assert go(*(4, 4, 6, 6) * 8) <= 4          # from either of the two buffer parities
    for ctx in (a, b):
        ctx.set_option(L.OPT_GRAPH_STEPS, 64)  # drops the graphs
    assert go(*[n for n in range(2, 40, 2) for _ in range(2)]) == 4
    assert go(*(40,) * 15) == 0
    assert go(*(40,) * 3) == 1                 # left sixteen times in a row: in place of the oldest
    assert go(*(2, 2, 2)) == 0                 # the oldest was 2
    assert go(8, 8, 8) == 0                    # still there
    np.testing.assert_allclose(a.read_populations(), b.read_populations(), rtol=0, atol=1e-12)
    np.testing.assert_allclose(a.read_capsule(1)[0], b.read_capsule(1)[0], rtol=0, atol=1e-11)
    assert b.capture_count == 0


def test_a_captured_caller_gets_plain_launches(L):
    import torch

    case = rows(2, 40, 200, 60, 8.0)
    s = torch.cuda.Stream()
    a, b = L.from_case(case, storage="fp64", stream=s), L.from_case(case, storage="fp64")
    for _ in range(3):
        for ctx in (a, b):
            ctx.step(4, o.DYNAMIC)
    a.sync()
    captured = a.capture_count
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        a.step(4, o.DYNAMIC)
        a.step(4, o.DYNAMIC)
    g.replay()
    torch.cuda.synchronize()
    b.step(8, o.DYNAMIC)
    assert a.capture_count == captured
    np.testing.assert_allclose(a.read_populations(), b.read_populations(), rtol=0, atol=1e-12)


@pytest.mark.parametrize("mode", ["global", "thread_local"])
def test_steps_beside_a_capture_of_another_stream(L, mode):
    # a rest that becomes a graph while the caller captures a stream the context does not use
    import torch

    case = rows(2, 40, 200, 60, 8.0)
    a, b = L.from_case(case, storage="fp64"), L.from_case(case, storage="fp64")
    s = torch.cuda.Stream()
    x = torch.zeros(1000, device="cuda")
    torch.cuda.synchronize()
    before = a.capture_count
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode=mode):
        x.add_(1.0)
        for _ in range(3):
            a.step(6, o.DYNAMIC)
        a.step(70, o.DYNAMIC)
        x.add_(1.0)
    assert a.capture_count - before == 2
    g.replay()
    torch.cuda.synchronize()
    for n in (6, 6, 6, 70):
        b.step(n, o.DYNAMIC)
    assert (x == 2.0).all()
    np.testing.assert_allclose(a.read_populations(), b.read_populations(), rtol=0, atol=1e-12)
