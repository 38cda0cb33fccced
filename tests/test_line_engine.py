"""The line transforms of P = 2^k and 3 * 2^k <= 768 (two or three stages) and the forms built on them.

CPU: a NumPy model of the stages, index for index as the kernels have them, equals the DFT for
every length, and its shared-memory accesses are free of bank conflicts.  GPU: single propagations
of every length against FP64, and gradients at the edges of the n = P/2 form (sides next to P/2,
boxes that leave the middle half P/4 .. 3P/4 on some angles) against the oracle."""

import numpy as np
import pytest

import holo_synth as hs

LENGTHS = [1 << k for k in range(4, 13)] + [48, 96, 192, 384, 768]


def shape(P):
    E = 48 if P % 3 == 0 else 32 if P >= 512 else 16
    T = P // E
    R = T // E if T > E else 1
    return E, T, R, (T + 1 if R > 1 else T + 2)


@pytest.mark.parametrize("P", LENGTHS)
def test_stages_equal_the_dft(P):
    E, T, R, _ = shape(P)
    x = np.random.default_rng(P).standard_normal((P, 2)) @ [1, 1j]
    A = np.fft.fft(x.reshape(E, T).T, axis=1)                 # [t][k1]: stage 1 of thread t
    X = np.empty(P, complex)
    for t in range(T):
        if R == 1:
            for k1 in range(t, E, T):                         # the thread's rows
                w = np.exp(-2j * np.pi * k1 / P)
                y = np.fft.fft(A[:, k1] * w ** np.arange(T))
                X[k1 + E * np.arange(T)] = y
        else:
            k1, u1 = t % E, t // E
            w2 = np.exp(-2j * np.pi * k1 / (E * E))
            B = np.stack([np.fft.fft(A[u::R, k1] * w2 ** np.arange(E)) for u in range(R)])
            for i in range(E // R):
                w3 = np.exp(-2j * np.pi * (t + T * i) / P)
                y = np.fft.fft(B[:, u1 + R * i] * w3 ** np.arange(R))
                X[t + T * (i + E // R * np.arange(R))] = y    # registers i + (E/R) k3
    assert np.linalg.norm(X - np.fft.fft(x)) < 1e-9 * np.linalg.norm(X)


@pytest.mark.parametrize("P,C,pitch", [(4096, 1, 0), (4096, 2, 8), (2048, 1, 0), (2048, 4, 4),
                                       (1024, 1, 0), (1024, 4, 4)])
def test_exchanges_are_free_of_bank_conflicts(P, C, pitch):
    """Lanes t * C + g of one warp (g the column of a column pass, lines `pitch` entries past
    their size): 8-byte accesses by half warps, 16-byte reads by quarter warps."""
    E, T, R, RS = shape(P)
    LS = E * RS + pitch

    def clean(addr, words, group):
        for w0 in range(0, T * C, 32):
            for l0 in range(w0, w0 + 32, group):
                banks = set()
                for lane in range(l0, l0 + group):
                    a = 2 * (addr(lane // C) + LS * (lane % C))
                    banks |= {(a + i) % 32 for i in range(words)}
                if len(banks) != group * words:
                    return False
        return True

    assert clean(lambda t: 5 * RS + t, 2, 16)                          # exchange 1, writes
    if R == 1:
        assert clean(lambda t: t * RS + 6, 4, 8)                       # rows, two values a read
    else:
        assert clean(lambda t: t % E * RS + t // E + R * 3, 2, 16)     # rows, and exchange 2 writes
        assert clean(lambda t: t % E * RS + t // E * R + 2 * R * R + 1, 2, 16)


gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("P", LENGTHS)
def test_propagation_error(P):
    """A transform pair is 2 log2 P levels, each adding about half an ulp (6e-8) of random
    rounding to a value, twice that where 2 a - s carries the error of s: 1.2e-7 sqrt(4 * 12) =
    8.3e-7 for rows and columns of P = 4096."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from oracle import holo as oh
    from paper_2407_20304_gb300 import Holo
    g = hs.WORKLOAD_GEOMETRY
    rng = np.random.default_rng(P)
    x = (rng.standard_normal((P, P)) + 1j * rng.standard_normal((P, P))).astype(np.complex64)
    h = Holo(max(16, P // 2), 1, 1, g["wavelength"], g["pixel"], g["Z"], g["z"][:1], pad=P)
    got = h.propagate(torch.from_numpy(x).cuda(), 3.1e-4).cpu().numpy()
    ref = oh.propagate(x.astype(np.complex128), 3.1e-4, g["wavelength"], g["pixel"])
    assert np.linalg.norm(got - ref) < 8.3e-7 * np.linalg.norm(ref)


@gpu
@pytest.mark.parametrize("n,P", [(30, 64), (32, 64), (64, 128), (66, 128), (128, 256), (256, 512),
                                 (512, 1024), (510, 1024), (1024, 2048),
                                 (24, 48), (48, 96), (96, 192), (192, 384), (384, 768), (386, 768)])
@pytest.mark.parametrize("shift", [0.0, 0.35])
def test_gradient_at_the_edges_of_the_half_form(n, P, shift):
    """shift * n pixels move the second angle's boxes out of the middle half."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from test_gpu_parity import dev, make_holo, make_problem, rel
    from oracle import holo as oh
    pr = make_problem(n, P, 2, J=2, seed=17 * n + P, point="object")
    pr["t"][1] += np.float32(shift * n)
    h = make_holo(pr)
    psi = dev(pr["psi"], torch.complex64)
    loss, gp, gq = h.gradient(psi)
    F, gp_ref, gq_ref = oh.gradients(pr["psi"], pr["q"], pr["t"], pr["sqrt_d"], pr["sqrt_dref"],
                                     pr["geo"])
    assert abs(h.forward(psi) - F) / F < 1e-5 and abs(loss - F) / F < 1e-5
    assert rel(gp.cpu().numpy(), gp_ref) < 1e-4 and rel(gq.cpu().numpy(), gq_ref) < 1e-4


@gpu
@pytest.mark.parametrize("n,P,J", [(64, 64, 3), (1024, 1024, 1), (62, 128, 8), (384, 768, 8)])
def test_gradient_without_padding_and_with_eight_distances(n, P, J):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from test_gpu_parity import dev, make_holo, make_problem, rel
    from oracle import holo as oh
    z = tuple(4.6e-4 + 0.5e-4 * j for j in range(J))
    pr = make_problem(n, P, 3, J=J, z=z, seed=5 * n + J, point="object")
    h = make_holo(pr)
    loss, gp, gq = h.gradient(dev(pr["psi"], torch.complex64))
    F, gp_ref, gq_ref = oh.gradients(pr["psi"], pr["q"], pr["t"], pr["sqrt_d"], pr["sqrt_dref"],
                                     pr["geo"])
    assert abs(loss - F) / F < 1e-5
    assert rel(gp.cpu().numpy(), gp_ref) < 1e-4 and rel(gq.cpu().numpy(), gq_ref) < 1e-4
