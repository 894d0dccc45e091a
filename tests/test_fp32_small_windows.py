"""FP32 operators at windows of few taps (``k_corr_one`` and the chunk groups of
``k_corr_warps`` in ``csrc/op_fp32.cu``) against the FP64 oracle.

Position counts around a block's 32, depths around the 16-deep chunks, the groups of 32
and 64 and the 128 elements of one staging, odd depths (rows off the 16-byte grid), and
scans large enough for the kernel of large problems.  Sums of at most 1e4 products in
three levels: below 1e-6.
"""
import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("win", [1, 3, 5, 7])
@pytest.mark.parametrize("px,py,nz,dz_um,nt", [(1, 1, 1, 10, 128), (31, 1, 5, 10, 128), (8, 4, 16, 10, 128), (11, 3, 33, 10, 160),
                                               (7, 9, 65, 2, 128), (5, 13, 129, 1, 128), (6, 6, 300, 0.5, 132), (160, 150, 4, 10, 128)])
def test_operators_match_oracle(win, px, py, nz, dz_um, nt):
    import torch

    import oracle
    from paper_2009_10173_gb300 import binding as B
    from paper_2009_10173_gb300 import configs, inputs
    from paper_2009_10173_gb300.model import Model
    cfg = configs.scaled(configs.TINY_32, px=px, py=py, nz=nz, nt=nt, win=win, n_patches=80, dz_m=dz_um * 1e-6,
                         z0_rel_m=-nz * dz_um * 0.5e-6)
    S = oracle.slab(cfg)
    m = Model(cfg, precision=B.OAM_PREC_FP32)
    H = inputs.gaussian(m.vol_shape, 61).astype(np.float32)
    s = inputs.gaussian(m.sig_shape, 62).astype(np.float32)
    f = m.forward(torch.from_numpy(H).cuda()).double().cpu().numpy()
    a = m.adjoint(torch.from_numpy(s).cuda()).double().cpu().numpy()
    m.close()
    for got, want in ((f, oracle.forward(S, H.astype(np.float64))), (a, oracle.adjoint(S, s.astype(np.float64)))):
        assert np.linalg.norm(want) > 0 and np.linalg.norm(got - want) <= 1e-6 * np.linalg.norm(want)
