"""What a position's error in the split-BF16 form is relative to.

The form takes the scan's y axis to the lateral frequency domain, so a position sees the
rounding of the transforms of the lines in its x window: an error of at most 1e-5 of its
own signal (three products of 22-bit terms and the accumulator's truncation) and 5e-7 of
the strongest (two FP32 line transforms of at most 512 points, 2^-22 of the terms) of
those lines, wherever on them it lies.  Lines outside the x window do not enter.
"""
import pytest

LOCAL, LINES = 1e-5, 5e-7


def pair(**over):
    from paper_2009_10173_gb300 import binding as B
    from paper_2009_10173_gb300 import configs
    from paper_2009_10173_gb300.model import Model
    cfg = configs.scaled(configs.VOLUME_200, nz=40, nt=512, win=15, n_patches=400, z0_rel_m=-100e-6, **over)
    return Model(cfg, precision=B.OAM_PREC_BF16X3), Model(cfg, precision=B.OAM_PREC_FP32)


@pytest.mark.gpu
@pytest.mark.parametrize("direction", ["forward", "adjoint"])
@pytest.mark.parametrize("ratio", [1.0, 1e-2, 1e-4, 1e-6])
def test_weak_rows_on_bright_lines(direction, ratio):
    """Bright and weak rows several windows apart on the same lines."""
    import torch
    m, ref = pair(px=24, py=150)
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn(m.vol_shape if direction == "forward" else m.sig_shape, generator=g, device="cuda")
    x[30:100] = 0
    x[100:] *= ratio
    got, want = getattr(m, direction)(x).double(), getattr(ref, direction)(x).double()
    m.close(), ref.close()
    weak = slice(110, 150)  # windows that hold weak rows alone
    err = (got - want)[weak].norm()
    assert err <= LOCAL * want[weak].norm() + LINES * want.norm()
    assert (got - want).norm() <= LOCAL * want.norm()


@pytest.mark.gpu
@pytest.mark.parametrize("direction", ["forward", "adjoint"])
@pytest.mark.parametrize("px", [120, 300])
@pytest.mark.parametrize("ratio", [1e-6, 1e-9, 1e-12])
def test_weak_columns_beside_bright_ones(direction, px, ratio):
    """Weak columns more than a window away from bright ones, also in the same block of positions."""
    import torch
    m, ref = pair(px=px, py=20)
    g = torch.Generator(device="cuda").manual_seed(8)
    x = torch.randn(m.vol_shape if direction == "forward" else m.sig_shape, generator=g, device="cuda")
    x[:, 40:] *= ratio
    got, want = getattr(m, direction)(x).double(), getattr(ref, direction)(x).double()
    m.close(), ref.close()
    weak = slice(48, None)
    assert (got - want)[:, weak].norm() <= LOCAL * want[:, weak].norm()
