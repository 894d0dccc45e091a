"""Tiles of the plain FP32 operators (``csrc/op_fp32.cu``).

On the CPU: for both position tilings, the staged strip holds the positions
x +- a of every lane and its padding is outside the grid.  On the GPU, against
the FP64 oracle at the FP32 operators' tolerance: sizes on both sides of the
rules that pick the kernel, the blocks per tile (one to eight, more than there
are row offsets in a share), the tiling and the tap table's place, odd depth
counts (scalar loads), partial output tiles and taps beyond the grid.
"""
import numpy as np
import pytest

MAX_STRIP = {32: 352, 128: 400}  # positions per block: longest strip of run-on tiles


def tiling(px, R, M):
    wrap = M + ((px + M - 2) // px + 2) * R
    return (px, wrap) if wrap <= MAX_STRIP[M] else ((px + M - 1) // M * M, M + 2 * R)


@pytest.mark.parametrize("px,py,R", [(1, 9, 5), (3, 40, 30), (32, 32, 5), (70, 37, 7), (127, 5, 30), (200, 7, 30),
                                     (129, 4, 127), (256, 3, 30), (17, 60, 1), (40, 40, 0)])
@pytest.mark.parametrize("M", [32, 128])
def test_strips_hold_every_tap(px, py, R, M):
    sp, strip = tiling(px, R, M)
    wp = px + R
    assert strip <= MAX_STRIP[M] and (sp == px or sp % M == 0)
    for t in range((py * sp + M - 1) // M):
        y0, x0 = t * M // sp, t * M % sp
        r = np.arange(strip)
        q = y0 * wp + x0 - R + r
        row, col = np.where(q < 0, -1, q // wp), np.where(q < 0, -1, q % wp)
        col = np.where(col < px, col, -1)
        m = np.arange(M)
        o = t * M + m
        y, x = o // sp, o % sp
        pm = (y - y0) * wp + (x - x0) + R
        out = (x < px) & (y < py)
        for a in (-R, -1, 0, 1, R):
            if abs(a) > R:
                continue
            i = pm + a
            assert i.min() >= 0 and i.max() < strip
            inside = out & (x + a >= 0) & (x + a < px)
            assert np.array_equal(col[i][inside], (x + a)[inside]) and np.array_equal(row[i][inside], y[inside])
            assert (col[i][out & ~inside] == -1).all()


@pytest.mark.gpu
@pytest.mark.parametrize("over", [
    dict(px=3, py=40, win=61, nz=13, nt=256, dx_m=4e-6, dy_m=4e-6), dict(px=150, py=90, win=7, nz=51, nt=192),
    dict(px=64, py=66, win=9, nz=47, nt=188), dict(px=33, py=5, win=5, nz=3, nt=128),
    dict(px=32, py=32, win=11, nz=48, nt=192), dict(px=70, py=37, win=15, nz=52, nt=200), dict(px=131, py=160, win=3, nz=33, nt=160), dict(px=260, py=190, win=5, nz=6, nt=128), dict(px=20, py=12, win=71, nz=17, nt=256, dx_m=4e-6, dy_m=4e-6), dict(px=9, py=3, win=21, nz=16, nt=192, dx_m=8e-6, dy_m=12e-6)],
    ids=lambda o: "x".join(str(o[k]) for k in ("px", "py", "win", "nz", "nt")))
def test_tiles_match_oracle(over):
    import torch

    import oracle
    from paper_2009_10173_gb300 import binding as B
    from paper_2009_10173_gb300 import configs, inputs
    from paper_2009_10173_gb300.model import Model
    cfg = configs.scaled(configs.TINY_32, n_patches=200, **over)
    S = oracle.slab(cfg)
    m = Model(cfg, precision=B.OAM_PREC_FP32)
    H = inputs.gaussian(m.vol_shape, 5).astype(np.float32)
    s = inputs.gaussian(m.sig_shape, 6).astype(np.float32)
    f = m.forward(torch.from_numpy(H).cuda()).double().cpu().numpy()
    a = m.adjoint(torch.from_numpy(s).cuda()).double().cpu().numpy()
    m.close()
    for got, want in ((f, oracle.forward(S, H.astype(np.float64))), (a, oracle.adjoint(S, s.astype(np.float64)))):
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
