"""The vector operations of a step on lengths and addresses that take the 16-byte and the 8-byte
forms: odd and even counts, slices that start on an odd element, fewer elements than a block."""

import numpy as np
import pytest

import holo_synth as hs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,off", [(1, 0), (2, 0), (2, 1), (31, 0), (4096, 1), (4097, 0),
                                   (65536, 0), (65538, 1), (1000002, 0)])
def test_vector_operations(n, off):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2407_20304_gb300 import Holo
    g = hs.WORKLOAD_GEOMETRY
    h = Holo(16, 1, 1, g["wavelength"], g["pixel"], g["Z"], g["z"][:1], pad=32)
    rng = np.random.default_rng(n + off)
    v = [(rng.standard_normal(n + off) + 1j * rng.standard_normal(n + off)).astype(np.complex64)
         for _ in range(4)]
    x, eta, gr, gp = (torch.from_numpy(a).cuda()[off:] for a in v)
    x64, eta64, gr64, gp64 = (a[off:].astype(np.complex128) for a in v)
    # sums of 2 n products: FP32 over 16 complex values (32 roundings of 6e-8 at most), then FP64
    dots = [(gr64, gr64), (gr64, eta64), (gp64, eta64)]
    size = [np.sum(np.abs(a) * np.abs(b)) for a, b in dots]
    ref = [np.vdot(a, b).real for a, b in dots]
    for got, r, s in zip(h.dy_dots(gr, gp, eta), ref, size):
        assert abs(got - r) <= 32 * 6e-8 * s
    assert abs(h.dot(gp, eta) - ref[2]) <= 32 * 6e-8 * size[2]
    e1, x1, e2, x2 = eta.clone(), x.clone(), eta.clone(), x.clone()
    h.direction(e1, gr, 0.37)
    h.step(x1, e1, -0.25)
    h.direction_step(x2, e2, gr, 0.37, -0.25)
    assert torch.equal(e1, e2) and torch.equal(x1, x2)
    ref_e = np.float32(0.37).astype(np.float64) * eta64 - gr64
    assert np.abs(e1.cpu().numpy() - ref_e).max() <= 4e-7 * np.abs(ref_e).max()
    assert np.abs(x1.cpu().numpy() - (x64 - 0.25 * ref_e)).max() <= 4e-7 * np.abs(x64).max() + 4e-7
    h.direction_step(x, eta, gr, 0.37, -0.25, dy=True)
    assert torch.equal(x, x1) and torch.equal(eta, e1)
    s = np.sum(np.abs(gr64) * np.abs(ref_e))
    assert abs(h.read_dy()[2] - np.vdot(gr64, ref_e).real) <= 64 * 6e-8 * s
