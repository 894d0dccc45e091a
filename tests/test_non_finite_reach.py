"""How far a non-finite input reaches along the output's samples and depths.

A non-finite value at one depth (sample) spoils the samples (depths) that its slab
bands hold, rounded to the kernel's groups, and leaves the others of the same position
finite.  The lateral-FFT form spreads it over every position, and to the neighbour
channel that shares a complex line.
"""
import numpy as np
import pytest


def setup(prec, **over):
    import oracle
    from paper_2009_10173_gb300 import configs
    from paper_2009_10173_gb300.model import Model
    cfg = configs.scaled(configs.TINY_32, **{**dict(px=12, py=9, nz=96, nt=512, win=5, n_patches=200, dz_m=12e-6,
                                                    z0_rel_m=-96 * 6e-6), **over})
    return cfg, (oracle.slab(cfg) != 0).any((0, 1)), Model(cfg, precision=prec)  # [depth][sample]


@pytest.mark.gpu
@pytest.mark.parametrize("direction", ["forward", "adjoint"])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_fft_form_keeps_other_bands_finite(direction, value):
    import torch

    from paper_2009_10173_gb300 import binding as B
    cfg, meets, m = setup(B.OAM_PREC_FFT)
    if direction == "adjoint":
        meets = meets.T  # [input][output]
    n = np.flatnonzero(meets.any(1))
    for e in (int(n[len(n) // 4]), int(n[len(n) // 2])):
        x = torch.randn(m.vol_shape if direction == "forward" else m.sig_shape, device="cuda")
        x[4, 5, e] = value
        bad = (~torch.isfinite(getattr(m, direction)(x))).any(0).any(0).cpu().numpy()
        reach = np.zeros_like(bad)
        for i in range(max(0, e - 1), e + 2):  # the channel of the same complex line is e - 1 or e + 1
            if i < meets.shape[0] and meets[i].any():
                o = np.flatnonzero(meets[i])
                reach[max(0, o[0] - 8):o[-1] + 8] = True  # groups of four outputs, and a band's last rounding
        assert bad[meets[e]].all()
        assert not (bad & ~reach).any() and not reach.all()
    m.close()


@pytest.mark.gpu
@pytest.mark.parametrize("direction", ["forward", "adjoint"])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_split_form_keeps_other_bands(direction, value):
    """Positions outside the window are untouched; inside it, the outputs that the 32 channels
    around the value do not reach are those of the same input with a zero in its place."""
    import torch

    from paper_2009_10173_gb300 import binding as B
    cfg, meets, m = setup(B.OAM_PREC_BF16X3, px=20, py=30, win=9, nz=192, dz_m=8e-6, z0_rel_m=-192 * 4e-6, nt=768)
    op = getattr(m, direction)
    if direction == "adjoint":
        meets = meets.T
    n, partial = np.flatnonzero(meets.any(1)), False
    for e in (int(n[0]), int(n[len(n) // 2]), int(n[-1])):
        x = torch.randn(m.vol_shape if direction == "forward" else m.sig_shape, device="cuda")
        x[15, 8, e] = 0
        want = op(x).clone()
        x[15, 8, e] = value
        got = op(x)
        bad = ~torch.isfinite(got)
        window = torch.zeros_like(bad)
        window[11:20, 4:13] = True
        assert not (bad & ~window).any()
        here = bad[11:20, 4:13].any(0).any(0).cpu().numpy()
        o = np.flatnonzero(meets[max(0, e - 47):e + 48].any(0))
        reach = np.zeros_like(here)
        reach[max(0, o[0] - 48):o[-1] + 49] = True
        assert here[meets[e]].all() and not (here & ~reach).any()
        partial = partial or not reach.all()
        keep = ~bad
        assert torch.equal(got[keep], want[keep])
        x[15, 8, e] = 0  # nothing of the marks is left
        assert torch.equal(op(x), want)
    assert partial
    m.close()
