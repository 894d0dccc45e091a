"""Grids and loops of the solver's vector kernels (``csrc/solvers.cu``).

A reduction runs four blocks of 256 threads per SM, fewer when the vector has
fewer float4 groups, and takes two groups per thread and turn.  LSQR and FISTA
against the oracle's FP64 solvers at the image tolerance, with vectors of a few
groups, of exactly one group per thread of the full grid, just above, and of
two and a remainder.
"""
import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("px,py,nt", [(2, 3, 128), (64, 64, 152), (64, 64, 156), (64, 64, 308), (61, 67, 128)])
def test_solvers_match_oracle(px, py, nt):
    import torch

    import oracle
    from oracle import solvers
    from paper_2009_10173_gb300 import binding as B
    from paper_2009_10173_gb300 import configs, inputs
    from paper_2009_10173_gb300.model import Model
    cfg = configs.scaled(configs.TINY_32, px=px, py=py, nz=5, nt=nt, win=3, n_patches=200)
    S = oracle.slab(cfg)
    m = Model(cfg, precision=B.OAM_PREC_FP32)
    s = oracle.forward(S, inputs.gaussian(m.vol_shape, 71))
    s += 0.05 * np.abs(s).max() * inputs.gaussian(m.sig_shape, 72)
    s = s.astype(np.float32)
    A, AT = (lambda v: oracle.forward(S, v)), (lambda v: oracle.adjoint(S, v))
    x, _ = m.lsqr(torch.from_numpy(s).cuda(), 6)
    y, info = m.fista(torch.from_numpy(s).cuda(), 6, power_iters=3, lambda_rel=1e-3, nonneg=False)
    x, y = x.double().cpu().numpy(), y.double().cpu().numpy()
    m.close()
    want, _ = solvers.lsqr(A, AT, s.astype(np.float64), 6)
    assert np.linalg.norm(x - want) <= 1e-3 * np.linalg.norm(want)
    want = solvers.fista(A, AT, s.astype(np.float64), 6, info.lambda_, info.L, nonneg=False)
    assert np.linalg.norm(y - want) <= 1e-3 * np.linalg.norm(want)
