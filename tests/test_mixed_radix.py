"""Mixed-radix transform sizes (``csrc/fft_mixed.cuh``).

On the CPU: the list of sizes is read from the source; each P = R1 R2 schedule
(transform of R1, roots W_P^(i2 k1), transform of R2, natural order at both
ends) gives numpy's DFT, the shared slots are distinct and inside the shared
memory of the launch, and a half-warp's accesses fall in distinct banks.  On
the GPU: the lateral-FFT form at every size, at the largest grid that fits it
and one position less, against the FP64 oracle at the FP32 operators'
tolerance.
"""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_10173_gb300", "csrc")


def sizes():
    src = open(os.path.join(CSRC, "fft_mixed.cuh")).read()
    body = src[src.index("#define OAM_MIX_SIZES(X)"):src.index("constexpr int kMixMax")]
    return [tuple(int(v) for v in t) for t in re.findall(r"X\((\d+), (\d+), (\d+)\)", body)]


def test_sizes_are_even_sorted_products():
    s = sizes()
    assert len(s) >= 15 and [p for p, _, _ in s] == sorted({p for p, _, _ in s})
    for p, r1, r2 in s:
        assert p == r1 * r2 and p % 2 == 0
        for r in (r1, r2):
            while r > 1:
                assert r % 2 == 0 or r % 3 == 0 or r % 5 == 0
                r //= 2 if r % 2 == 0 else 3 if r % 3 == 0 else 5


@pytest.mark.parametrize("P,R1,R2", sizes())
def test_two_passes_compute_the_dft(P, R1, R2):
    rng = np.random.Generator(np.random.PCG64(P))
    x = rng.standard_normal(P) + 1j * rng.standard_normal(P)
    Y = np.fft.fft(x.reshape(R1, R2), axis=0)  # [k1][i2]
    Y *= np.exp(-2j * np.pi * np.outer(np.arange(R1), np.arange(R2)) / P)
    X = np.fft.fft(Y, axis=1)  # [k1][k2]
    got = np.empty(P, complex)
    got[np.add.outer(np.arange(R1), R1 * np.arange(R2))] = X
    want = np.fft.fft(x)
    assert np.allclose(got, want, atol=1e-12 * np.abs(want).max())


@pytest.mark.parametrize("P,R1,R2", sizes())
@pytest.mark.parametrize("KL", [8, 16])
def test_shared_slots(P, R1, R2, KL):
    rs = R2 * KL + (KL if KL < 16 else 0)
    slot = lambda k1, i2, l: k1 * rs + i2 * KL + l
    every = [slot(k, i, l) for k in range(R1) for i in range(R2) for l in range(KL)]
    assert len(set(every)) == P * KL and max(every) < R1 * rs
    items1 = [(i2, l) for i2 in range(R2) for l in range(KL)]  # pass 1 writes, pass 2 reads
    items2 = [(k1, l) for k1 in range(R1) for l in range(KL)]
    for h in range(0, len(items1) - 15, 16):
        assert len({slot(0, i, l) % 16 for i, l in items1[h:h + 16]}) == 16
    if (R2 + (1 if KL < 16 else 0)) % 2 or KL == 16:  # rows an odd number of half-rows apart
        for h in range(0, len(items2) - 15, 16):
            assert len({slot(k, 0, l) % 16 for k, l in items2[h:h + 16]}) == 16


@pytest.mark.gpu
@pytest.mark.parametrize("P,R1,R2", sizes())
def test_fft_form_at_every_size(P, R1, R2):
    import torch

    import oracle
    from paper_2009_10173_gb300 import binding as B
    from paper_2009_10173_gb300 import configs, inputs
    from paper_2009_10173_gb300.model import Model
    for side in {max(1, P - 1), max(1, P - 2)}:  # halo R = 1: need = side + 1
        for px, py in ((side, 3), (2, side)):
            cfg = configs.scaled(configs.TINY_32, px=px, py=py, nz=7, nt=128, win=3, n_patches=200)
            S = oracle.slab(cfg)
            m = Model(cfg, precision=B.OAM_PREC_FFT)
            H = inputs.gaussian(m.vol_shape, 41).astype(np.float32)
            s = inputs.gaussian(m.sig_shape, 42).astype(np.float32)
            f = m.forward(torch.from_numpy(H).cuda()).double().cpu().numpy()
            a = m.adjoint(torch.from_numpy(s).cuda()).double().cpu().numpy()
            m.close()
            for got, want in ((f, oracle.forward(S, H.astype(np.float64))), (a, oracle.adjoint(S, s.astype(np.float64)))):
                assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want), (px, py)
