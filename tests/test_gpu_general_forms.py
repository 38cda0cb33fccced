"""The passes' general forms (a side other than P/2, probe shifts) against the oracle: pass B with the
chirp in shared memory and, for tall boxes at P = 2048 and 4096, in global memory.  Tolerances as in
test_gpu_parity.py: loss 1e-5, gradients 1e-4 (relative L2)."""

import numpy as np
import pytest

import test_gpu_parity as plain
from oracle import holo as oh

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


def check(loss, gp, gq, ref):
    F, gp_ref, gq_ref = ref
    assert abs(loss - F) / F < plain.LOSS_TOL
    assert plain.rel(gp.cpu().numpy(), gp_ref) < plain.GRAD_TOL
    assert plain.rel(gq.cpu().numpy(), gq_ref) < plain.GRAD_TOL


# n = P/2 + 2 and sides on both sides of the longest box that keeps the chirp in shared memory
@pytest.mark.parametrize("n,P,K,J", [(514, 1024, 2, 3), (608, 2048, 2, 2), (768, 2048, 1, 2),
                                     (770, 2048, 1, 2), (1026, 2048, 1, 4), (608, 4096, 1, 2),
                                     (2050, 4096, 1, 2)])
@pytest.mark.parametrize("stage", [-1, 0])
def test_general_form_with_and_without_the_stage(n, P, K, J, stage):
    pr = plain.make_problem(n, P, K, J=J, seed=13 * n + J, point="object")
    h = plain.make_holo(pr)
    h.set_schedule(0, stage, -1)
    psi = plain.dev(pr["psi"], torch.complex64)
    loss_f = h.forward(psi)
    loss, gp, gq = h.gradient(psi)
    assert loss_f == loss
    check(loss, gp, gq, oh.gradients(pr["psi"], pr["q"], pr["t"], pr["sqrt_d"], pr["sqrt_dref"],
                                     pr["geo"]))
