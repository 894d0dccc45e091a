"""oam_model_bytes bounds the built split form where the planner's wider bands and the
build's bands choose different part counts (``choose_parts`` in ``csrc/op_tc.cu``): a
part's sums are the one buffer that a narrower support can make larger."""
import random

import pytest

# (px, py, nz, win, focal mm, aperture mm): the build takes more parts than the widened plan's own choice
SHAPES = [(161, 50, 75, 29, 5.8, 3.3), (111, 75, 77, 21, 3.3, 2.5), (205, 36, 41, 23, 4.2, 2.1),
          (57, 37, 55, 39, 3.954589, 3.324812)]


def draws():
    rng = random.Random(17)
    return [(rng.randrange(24, 220), rng.randrange(24, 120), rng.randrange(24, 120), 2 * rng.randrange(8, 24) - 1,
             rng.uniform(3, 6), rng.uniform(2, 4)) for _ in range(12)]


@pytest.mark.gpu
@pytest.mark.parametrize("px,py,nz,win,focal,aperture", SHAPES + draws())
def test_planned_bytes_bound_the_build(px, py, nz, win, focal, aperture):
    from paper_2009_10173_gb300 import binding as B
    from paper_2009_10173_gb300 import configs
    from paper_2009_10173_gb300.model import Model
    cfg = configs.scaled(configs.VOLUME_200, px=px, py=py, nz=nz, nt=1024, win=win, focal_m=focal * 1e-3,
                         aperture_m=aperture * 1e-3, n_patches=800, z0_rel_m=-(nz / 2) * 5e-6)
    planned = B.oam_model_bytes(cfg, B.OAM_PREC_BF16X3)
    m = Model(cfg, precision=B.OAM_PREC_BF16X3)
    built = m.info.device_bytes
    m.close()
    assert built <= planned, (built, planned)
