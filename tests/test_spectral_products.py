"""Spectral products of the lateral-FFT form (``k_fft_apply`` in
``csrc/op_fft.cu``): both directions against the FP64 oracle at the FP32
operators' tolerance, at depth counts around the kernel's four-output groups,
its 16-element steps and its 32-output windows, with sample supports that start
off a group's boundary, and at one more and one fewer warp than windows.
"""
import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("nz", [1, 3, 4, 5, 15, 16, 17, 31, 32, 33, 63, 65, 129, 161])
def test_products_match_oracle(nz):
    import torch

    import oracle
    from paper_2009_10173_gb300 import binding as B
    from paper_2009_10173_gb300 import configs, inputs
    from paper_2009_10173_gb300.model import Model
    cfg = configs.scaled(configs.TINY_32, px=6, py=5, nz=nz, nt=512, win=5, n_patches=200)
    S = oracle.slab(cfg)
    m = Model(cfg, precision=B.OAM_PREC_FFT)
    H = inputs.gaussian(m.vol_shape, 51).astype(np.float32)
    s = inputs.gaussian(m.sig_shape, 52).astype(np.float32)
    f = m.forward(torch.from_numpy(H).cuda()).double().cpu().numpy()
    a = m.adjoint(torch.from_numpy(s).cuda()).double().cpu().numpy()
    m.close()
    for got, want in ((f, oracle.forward(S, H.astype(np.float64))), (a, oracle.adjoint(S, s.astype(np.float64)))):
        assert np.linalg.norm(want) > 0 and np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
