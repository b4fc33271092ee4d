"""Batched FP16 cases repeat themselves: rings of one warp add their force shares in a fixed
order, which FP16 storage needs (a share added in another order moves populations by storage
steps)."""
import numpy as np
import pytest

from paper_1903_03356_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_fp16_batches_repeat_bit_for_bit():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_03356_gb300 import lbmib as L
    cases = [W.shear_capsule(50, 50, radius=5.0037, n=32, ca=10.0 ** (-2.2 + 0.02 * k), scheme=W.KINEMATIC,
                             centre=(25.1137 + 0.007 * k, 24.5929)) for k in range(24)]
    out = []
    for _ in range(3):
        b = L.Batch(cases, storage="fp16")
        b.step(300)
        out.append((b.observables(), np.stack([b.read_capsule(k)[0] for k in range(24)]),
                    np.stack([b.read_populations(k) for k in range(24)])))
        b.close()
    for other in out[1:]:
        for x, y in zip(out[0], other):
            np.testing.assert_array_equal(x, y)
