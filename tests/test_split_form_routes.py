"""Where the split-BF16 form sums by the FP32 kernels (``uses_direct`` in
``csrc/op_fp32.cu``) and where by its line transforms: both against the FP64 oracle, on
both sides of the rule (windows of one tap, few taps and few or many positions, single
rows, the first windows beyond nine folded taps), with lines in several segments.
"""
import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("px,py,win,nz,direct", [
    (13, 9, 1, 20, True), (200, 180, 1, 9, True), (1, 1, 1, 5, True), (16, 16, 3, 20, True), (12, 10, 5, 33, True),
    (40, 1, 11, 9, True), (40, 1, 17, 9, True), (1, 40, 17, 9, True), (40, 1, 19, 9, False), (6, 3, 7, 9, False),
    (230, 200, 3, 20, False), (33, 1, 31, 9, False), (4, 511, 7, 9, False), (5, 520, 9, 9, False),
    (7, 600, 11, 9, False)])
def test_both_sides_match_oracle(px, py, win, nz, direct):
    import torch

    import oracle
    from paper_2009_10173_gb300 import binding as B
    from paper_2009_10173_gb300 import configs, inputs
    from paper_2009_10173_gb300.model import Model
    cfg = configs.scaled(configs.TINY_32, px=px, py=py, win=win, nz=nz, nt=160, n_patches=200)
    S = oracle.slab(cfg)
    planned = B.oam_model_bytes(cfg, B.OAM_PREC_BF16X3)
    m = Model(cfg, precision=B.OAM_PREC_BF16X3)
    assert m.info.device_bytes <= planned
    assert (m.info.exec_flops_forward == 0) == direct == (m.info.exec_flops_adjoint == 0)
    H = inputs.gaussian(m.vol_shape, 91).astype(np.float32)
    s = inputs.gaussian(m.sig_shape, 92).astype(np.float32)
    f = m.forward(torch.from_numpy(H).cuda()).double().cpu().numpy()
    a = m.adjoint(torch.from_numpy(s).cuda()).double().cpu().numpy()
    m.close()
    tol = 1e-6 if direct else 2e-5
    for got, want in ((f, oracle.forward(S, H.astype(np.float64))), (a, oracle.adjoint(S, s.astype(np.float64)))):
        assert np.linalg.norm(want) > 0 and np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
