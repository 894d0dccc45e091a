"""LSQR and FISTA against the FP64 solvers at a few steps, to the operators' precision.

An FP32 operator is within 1e-6 of the oracle's; six steps apply twelve, and on these
well-conditioned problems each passes its error on about once: 1.2e-5, below 2e-5.  The
image tolerance of 1e-3 would let a wrong low-order coefficient pass.
"""
import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["OAM_PREC_FP32", "OAM_PREC_FFT"])
@pytest.mark.parametrize("px,py,nt,damp", [(2, 3, 128, 0.0), (64, 64, 152, 0.0), (61, 67, 128, 0.0), (33, 17, 160, 2.0)])
def test_solvers_to_operator_precision(form, px, py, nt, damp):
    import torch

    import oracle
    from oracle import solvers
    from paper_2009_10173_gb300 import binding as B
    from paper_2009_10173_gb300 import configs, inputs
    from paper_2009_10173_gb300.model import Model
    cfg = configs.scaled(configs.TINY_32, px=px, py=py, nz=5, nt=nt, win=3, n_patches=200)
    S = oracle.slab(cfg)
    m = Model(cfg, precision=getattr(B, form))
    s = oracle.forward(S, inputs.gaussian(m.vol_shape, 81))
    s += 0.05 * np.abs(s).max() * inputs.gaussian(m.sig_shape, 82)
    s = s.astype(np.float32)
    A, AT = (lambda v: oracle.forward(S, v)), (lambda v: oracle.adjoint(S, v))
    x, _ = m.lsqr(torch.from_numpy(s).cuda(), 6, damp=damp)
    y, info = m.fista(torch.from_numpy(s).cuda(), 6, power_iters=3, lambda_rel=1e-3)
    x, y = x.double().cpu().numpy(), y.double().cpu().numpy()
    m.close()
    want, _ = solvers.lsqr(A, AT, s.astype(np.float64), 6, damp=damp)
    assert np.linalg.norm(x - want) <= 2e-5 * np.linalg.norm(want)
    want = solvers.fista(A, AT, s.astype(np.float64), 6, info.lambda_, info.L, nonneg=True)
    assert np.linalg.norm(y - want) <= 2e-5 * np.linalg.norm(want)
