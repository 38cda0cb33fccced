"""The split of pass B's partial last round.

CPU: the rules of csrc/holo_split.h, compiled as they are: no more blocks than items, every item in
exactly one block, every partial sum found by the combine kernel's run of blocks and slots.  GPU:
problems of few and of many (column group, plane) items against the oracle, repeats bit for bit."""

import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2407_20304_gb300", "csrc")
WRAP = """
#include "holo_split.h"
extern "C" {
int form(int sched, int groups, int full) { return holo::split_form(sched, groups, full); }
int blocks(int full, int sms, long long items) { return holo::split_blocks(full, sms, items); }
long long begin(long long t, int nblk, int b) { return holo::split_begin(t, nblk, b); }
int slots(long long t, int nblk, long long per) { return holo::split_slots(t, nblk, per); }
void run(long long t, int nblk, long long per, int tg, int* out) {
  const holo::SplitRun r = holo::split_run(t, nblk, per, tg);
  out[0] = r.first; out[1] = r.last; out[2] = r.slot;
}
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("split")
    (d / "wrap.cpp").write_text(WRAP)
    subprocess.run([cxx, "-shared", "-fPIC", "-std=c++17", "-I", CSRC, str(d / "wrap.cpp"), "-o",
                    str(d / "wrap.so")], check=True)
    lib = ctypes.CDLL(str(d / "wrap.so"))
    lib.begin.restype = ctypes.c_longlong
    lib.begin.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    lib.blocks.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_longlong]
    lib.slots.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_longlong]
    lib.run.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_longlong, ctypes.c_int,
                        ctypes.POINTER(ctypes.c_int)]
    return lib


@pytest.mark.parametrize("full", [152, 304, 608, 760])
def test_blocks_follow_the_items(rules, full):
    for items in list(range(1, 700)) + [1216, 5000, 10 ** 6, 10 ** 9]:
        b = rules.blocks(full, 152, items)
        assert 1 <= b <= min(items, full)
        # every SM has work where there is enough of it, and blocks share it two items at a time
        # only where every SM already has two blocks
        assert b >= min(items, 152)
        assert b == min(full, items) or b >= min(full, 304)


@pytest.mark.parametrize("full", [152, 304, 608])
def test_full_rounds_are_never_split(rules, full):
    """Form 1 gives up the Y stage: it must not be taken where no round is partial."""
    for sched in (-1, 0, 1, 2):
        for rounds in (1, 2, 5):
            assert rules.form(sched, rounds * full, full) == 0
            partial = rules.form(sched, rounds * full + 1, full)
            assert partial == (sched if sched >= 0 else (2 if rounds < 3 else 0))


@pytest.mark.parametrize("groups,per", [(1, 1), (1, 2), (1, 7), (1, 40), (2, 8), (5, 3), (13, 20),
                                        (33, 8), (152, 1), (153, 1), (305, 1), (305, 2), (306, 72),
                                        (609, 3), (700, 5)])
@pytest.mark.parametrize("full", [152, 304, 608])
def test_items_and_slots(rules, groups, per, full):
    nblk = rules.blocks(full, 152, groups * per)
    tail = groups % nblk
    t = tail * per
    slots = rules.slots(t, nblk, per)
    if not t:
        assert slots == 0
        return
    first = [rules.begin(t, nblk, b) for b in range(nblk + 1)]
    assert first[0] == 0 and first[-1] == t and all(x <= y for x, y in zip(first, first[1:]))
    parts = {g: [] for g in range(tail)}     # group -> (block, slot) in block order
    for b in range(nblk):
        if first[b] == first[b + 1]:
            continue
        g0, g1 = first[b] // per, (first[b + 1] - 1) // per
        assert g1 - g0 < slots
        for g in range(g0, g1 + 1):
            parts[g].append((b, g - g0))
    out = (ctypes.c_int * 3)()
    for g in range(tail):
        rules.run(t, nblk, per, g, out)
        lo, hi, slot = out
        found = [(b, slot if b == lo else 0) for b in range(lo, hi + 1) if first[b] < first[b + 1]]
        assert found == parts[g]


@pytest.mark.gpu
@pytest.mark.parametrize("n,P,K,J", [(32, 64, 1, 1), (32, 64, 1, 2), (32, 64, 7, 1), (32, 64, 10, 4),
                                     (40, 64, 5, 3), (100, 256, 5, 4), (128, 256, 9, 4),
                                     (258, 512, 2, 4)])
def test_gradient_of_few_and_many_items(n, P, K, J):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from oracle import holo as oh
    from test_gpu_parity import GRAD_TOL, LOSS_TOL, dev, make_holo, make_problem, rel
    pr = make_problem(n, P, K, J=J, seed=3 * n + K, point="object")
    h = make_holo(pr)
    psi = dev(pr["psi"], torch.complex64)
    loss, gp, gq = h.gradient(psi)
    F, gp_ref, gq_ref = oh.gradients(pr["psi"], pr["q"], pr["t"], pr["sqrt_d"], pr["sqrt_dref"],
                                     pr["geo"])
    assert abs(loss - F) / F < LOSS_TOL
    assert rel(gp.cpu().numpy(), gp_ref) < GRAD_TOL and rel(gq.cpu().numpy(), gq_ref) < GRAD_TOL
    loss2, gp2, gq2 = h.gradient(psi)
    assert loss2 == loss and torch.equal(gp2, gp) and torch.equal(gq2, gq)
