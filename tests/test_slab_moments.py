"""Slab bands from patch moments (``k_slab_moments`` in ``csrc/slab.cu``).

Against the FP64 oracle at the slab's tolerance: patch counts around the
kernel's warps, segments and chunks, voxels near the focus (all arrivals in a
few samples) and far from it, truncations whose edge falls on, just below and
just above half a sample, and pulses that the polynomials do not reach (a
carrier near the Nyquist rate, a truncation below two samples), which take the
direct sum.
"""
import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("over", [
    dict(n_patches=8), dict(n_patches=40), dict(n_patches=1016), dict(n_patches=1032), dict(n_patches=2056),
    dict(nz=1, z0_rel_m=0.0, win=1), dict(trunc_sigma=3.0), dict(trunc_sigma=4.485), dict(trunc_sigma=4.49),
    dict(trunc_sigma=1.0), dict(trunc_sigma=0.6), dict(fc_hz=110e6, frac_bw=0.8), dict(fc_hz=12e6)],
    ids=lambda o: "-".join("%s_%g" % kv for kv in o.items()))
def test_columns_match_oracle(over):
    import oracle
    from paper_2009_10173_gb300 import binding as B
    from paper_2009_10173_gb300 import configs
    from paper_2009_10173_gb300.model import Model
    cfg = configs.scaled(configs.TINY_32, **{**dict(px=4, py=4, nz=9, nt=512, win=5), **over})
    S = oracle.slab(cfg)
    m = Model(cfg, precision=B.OAM_PREC_FP32)
    R = (cfg["win"] - 1) // 2
    got = np.zeros_like(S)
    for b in range(-R, R + 1):
        for a in range(-R, R + 1):
            for k in range(cfg["nz"]):
                got[b + R, a + R, k] = m.slab_column(b, a, k).double().cpu().numpy()
    m.close()
    assert np.linalg.norm(got - S) <= 1e-6 * np.linalg.norm(S)
