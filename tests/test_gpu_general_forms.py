"""The passes' general forms (a side other than P/2, probe shifts) against the oracle: pass B with the
chirp in shared memory and, for tall boxes at P = 2048 and 4096, in global memory; and the batch of
problems of one line length whose general forms share their launches.  Tolerances as in
test_gpu_parity.py: loss 1e-5, gradients 1e-4 (relative L2)."""

import numpy as np
import pytest

import test_gpu_parity as plain
import test_gpu_probe_shift as shifted
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


def test_batch_of_shifted_and_unshifted_problems():
    """Problems of one line length, with and without probe shifts, staged and not, in one batch:
    every problem's results are those of its own calls bit for bit and match the oracle.  (With
    probe shifts the reference field is part of the full-grid rows; added in pass B once more it
    made the results of such a batch wrong.)"""
    from paper_2407_20304_gb300.batch import HoloBatch, Instance
    insts, refs = [], []
    for i, (n, P, K, J, ps) in enumerate([(64, 128, 3, 2, True), (64, 128, 2, 4, False),
                                          (50, 128, 3, 3, False), (96, 192, 2, 2, True),
                                          (72, 192, 2, 2, False), (128, 128, 2, 1, True),
                                          (514, 1024, 1, 2, False), (512, 1024, 1, 2, True),
                                          (608, 2048, 1, 1, False), (1026, 2048, 1, 2, False)]):
        mod = shifted if ps else plain
        pr = mod.make_problem(n, P, K, J=J, seed=100 + i, point="object")
        h = mod.make_holo(pr, chunk=min(2, K))
        kw = {"probe_shifts": pr["s"]} if ps else {}
        refs.append(oh.gradients(pr["psi"], pr["q"], pr["t"], pr["sqrt_d"], pr["sqrt_dref"],
                                 pr["geo"], **kw))
        insts.append(Instance(h, plain.dev(pr["psi"], torch.complex64),
                              plain.dev(pr["q"], torch.complex64)))
    b = HoloBatch(insts)
    b.prepare_persistent()
    b.run_loop()
    torch.cuda.synchronize()
    own = [(it.h.read_loss(), it.grad_psi.clone(), it.grad_q.clone()) for it in b.inst]
    for it in b.inst:
        it.grad_psi.fill_(float("nan"))
        it.grad_q.fill_(float("nan"))
    b.capture_persistent()
    b.replay_persistent()
    torch.cuda.synchronize()
    for it, (loss, gp, gq), ref in zip(b.inst, own, refs):
        assert it.h.read_loss() == loss
        assert torch.equal(it.grad_psi, gp) and torch.equal(it.grad_q, gq)
        check(loss, gp, gq, ref)
    b.close()


@pytest.mark.parametrize("n,P,K,J", [(512, 1024, 2, 2), (700, 1024, 3, 1), (768, 1536, 1, 2),
                                     (1024, 2048, 1, 2), (1200, 4096, 2, 1)])
@pytest.mark.parametrize("stage", [-1, 0])
def test_probe_shifts_with_and_without_the_stage(n, P, K, J, stage):
    pr = shifted.make_problem(n, P, K, J=J, seed=19 * n + J, point="object")
    h = shifted.make_holo(pr)
    h.set_schedule(0, stage, -1)
    psi = plain.dev(pr["psi"], torch.complex64)
    loss_f = h.forward(psi)
    loss, gp, gq = h.gradient(psi)
    assert loss_f == loss
    check(loss, gp, gq, oh.gradients(pr["psi"], pr["q"], pr["t"], pr["sqrt_d"], pr["sqrt_dref"],
                                     pr["geo"], probe_shifts=pr["s"]))
    h.set_probe_shifts(None)  # back to the boxes: the stage's tensor map and sizes follow
    loss_b = h.forward(psi)
    u = oh.gradients(pr["psi"], pr["q"], pr["t"], pr["sqrt_d"], pr["sqrt_dref"], pr["geo"])[0]
    assert abs(loss_b - u) / u < plain.LOSS_TOL
