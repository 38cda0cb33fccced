"""Errors of a propagation at every line length, the coherent part apart from the random one.

A propagation is four transforms and two chirps per element (rows, columns).  Rounding to nearest
leaves a random error, 1.2e-7 sqrt(4 log2 P) (a transform pair per axis is 2 log2 P levels of about
1.2e-7 each).  Twiddle constants rounded to FP32 are no longer of length one: each transform scales
all values by the same factor, 1 - 7.3e-8 at P = 4096, which the chirp tables take out again.  Left in,
it would be 2.9e-7 of a propagation at P = 4096; what may remain (twiddle and chirp tables, whose
roundings average out over their entries) is below a third of that."""

import numpy as np
import pytest

import holo_synth as hs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("P", [1 << k for k in range(4, 13)] + [3 << k for k in range(4, 11)])
def test_coherent_and_random_error(P):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from oracle import holo as oh
    from paper_2407_20304_gb300 import Holo
    g = hs.WORKLOAD_GEOMETRY
    rng = np.random.default_rng(P)
    x = (rng.standard_normal((P, P)) + 1j * rng.standard_normal((P, P))).astype(np.complex64)
    h = Holo(max(16, P // 2), 1, 1, g["wavelength"], g["pixel"], g["Z"], g["z"][:1], pad=P)
    got = h.propagate(torch.from_numpy(x).cuda(), 4.6e-4).cpu().numpy().astype(np.complex128)
    ref = oh.propagate(x.astype(np.complex128), 4.6e-4, g["wavelength"], g["pixel"])
    nn = np.vdot(ref, ref).real
    scale = np.vdot(ref, got).real / nn - 1.0
    print(f"P={P}: scale {scale:.2e}, error {np.linalg.norm(got - ref) / np.sqrt(nn):.2e}")
    assert abs(scale) < 1e-7
    assert np.linalg.norm(got - ref) < 1.2e-7 * np.sqrt(4 * np.log2(P)) * np.sqrt(nn)
