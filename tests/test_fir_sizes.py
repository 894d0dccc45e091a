"""Mixed-radix filter sizes (``k_fir_mixed`` in ``csrc/op_filter.cu``).

On the CPU: the sizes are read from the source; the three passes with the
spectrum stored where the forward transform leaves it give the circular
convolution, and the shared slots are distinct and inside the launch's memory.
On the GPU: at the largest and the least length that picks each size, with line
counts that leave a block's line pair partly empty, against the direct FP64
sum.  An FP32 transform pair of N points errs by about 2 log2(N) 2^-24 of the
signal's norm, 1.4e-6 at 4096.
"""
import os
import re

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_10173_gb300", "csrc",
                   "op_filter.cu")


def sizes():
    src = open(SRC).read()
    body = src[src.index("#define OAM_FIR_SIZES(X)"):src.index("constexpr int fir_threads")]
    return [tuple(int(v) for v in t) for t in re.findall(r"X\((\d+), (\d+), (\d+), (\d+)\)", body)]


@pytest.mark.parametrize("N,A,B,C", sizes())
def test_passes_compute_the_convolution(N, A, B, C):
    assert N == A * B * C and C % 8 == 0
    M, f = B * C, np.arange(N)
    slots = [i + i // 8 for i in range(N)]
    assert len(set(slots)) == N and max(slots) < N + N // 8
    rng = np.random.Generator(np.random.PCG64(N))
    x = rng.standard_normal(N) + 1j * rng.standard_normal(N)
    taps = rng.standard_normal(N // 4)
    h = np.concatenate([taps, np.zeros(N - 2 * len(taps) + 1), taps[:0:-1]])
    H = np.fft.fft(h).real / N
    hb = np.empty(N)
    hb[(f % A * B + f // A % B) * C + f // (A * B)] = H
    W = lambda n, j: np.exp(-2j * np.pi * j / n)
    t1 = W(N, np.outer(np.arange(A), np.arange(M)))
    t2 = W(M, np.outer(np.arange(B), np.arange(C)))
    v = (np.fft.fft(x.reshape(A, M), axis=0) * t1).reshape(A, B, C)
    v = np.fft.fft(np.fft.fft(v, axis=1) * t2, axis=2) * hb.reshape(A, B, C)
    swap = lambda z: z.imag + 1j * z.real
    v = np.fft.fft(np.fft.fft(swap(v), axis=2) * t2, axis=1).reshape(A, M)
    got = swap(np.fft.fft(v * t1, axis=0)).reshape(N)
    want = np.fft.ifft(np.fft.fft(x) * np.fft.fft(h).real)
    assert np.allclose(got, want, atol=1e-11 * np.abs(want).max())


@pytest.mark.gpu
@pytest.mark.parametrize("need", sorted({n for s in sizes() for n in (s[0], s[0] + 1)} | {256, 257}))
def test_lengths_match_the_direct_sum(need):
    import torch

    from paper_2009_10173_gb300 import binding as B
    from paper_2009_10173_gb300 import configs, inputs
    from paper_2009_10173_gb300.model import Model
    nt = (need - need // 3) // 4 * 4
    L = need - nt
    for px, py in ((3, 3), (5, 2), (1, 4)):
        cfg = configs.scaled(configs.TINY_32, px=px, py=py, nz=2, nt=nt, win=1, n_patches=200)
        m = Model(cfg, precision=B.OAM_PREC_FP32)
        taps = np.array(B.oam_bandpass_taps(0.5e6, 80e6, cfg["fs_hz"], L))
        m.set_filter(taps)
        s = inputs.gaussian(m.sig_shape, need).astype(np.float32)
        got = m.filter_signals(torch.from_numpy(s).cuda()).double().cpu().numpy().reshape(-1, nt)
        m.close()
        h = np.concatenate([taps[:0:-1], taps])
        want = np.array([np.convolve(r, h)[L:L + nt] for r in s.astype(np.float64).reshape(-1, nt)])
        assert np.linalg.norm(got - want) <= 2e-6 * np.linalg.norm(want)
