"""The loss of a plane against its FP64 sum where FP32 additions would lose most of its terms.

A uniform probe through empty space gives u = 1 on every detector pixel.  The data put one term of
64^2 in the first crop row of every thread and terms of 5e-8 times that in its other rows: added to
the large one by one in FP32 each of them is lost, (rows - 1) * 5e-8 of the loss.  The kernel adds
the `rows` terms of a thread in groups of four: 3 + rows / 4 - 1 roundings of 2^-24 at most."""

import numpy as np
import pytest

import holo_synth as hs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# T: threads of a line, whose rows t + T c the registers c of thread t hold
@pytest.mark.parametrize("n,P,T", [(768, 768, 16), (384, 768, 16), (1024, 1024, 32),
                                   (512, 1024, 32), (256, 256, 16)])
def test_small_terms_beside_a_large_one(n, P, T):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2407_20304_gb300 import Holo
    g = hs.WORKLOAD_GEOMETRY
    h = Holo(n, 1, 1, g["wavelength"], g["pixel"], g["Z"], g["z"][:1], pad=P, w_ref=0.0)
    h.set_shifts(np.zeros((1, 1, 2), np.float32))
    d = np.full((1, 1, n, n), 1.0 + 64.0 * np.sqrt(5e-8), np.float32)
    d[:, :, :T] = 65.0
    h.set_data(torch.from_numpy(d).cuda())
    h.set_probe(torch.ones(P, P, dtype=torch.complex64, device="cuda"))
    psi = torch.ones(1, n, n, dtype=torch.complex64, device="cuda")
    ref = np.sum((1.0 - d.astype(np.float64)) ** 2)
    rows = n // T
    tol = (rows // 4 + 2) * 2.0 ** -24 + 2e-8   # 2e-8: u, whose error is 1e-7 of 64
    assert tol < (rows - 1) * 5e-8
    loss = h.gradient(psi)[0]
    assert abs(h.forward(psi) - ref) < tol * ref
    assert abs(loss - ref) < tol * ref
